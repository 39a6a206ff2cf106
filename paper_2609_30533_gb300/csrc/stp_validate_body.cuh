// Every-point edge validation (verdicts and clearances with no early exit: each
// check point of each edge is evaluated, also after a collision), and the pieces it shares
// with the bounded-motion validation in stp_edges_body.cuh: packed FP32
// arithmetic, obstacle interpolation, block scan.
//
// Mapping: a persistent grid walks windows of consecutive edges, one check point
// per lane; a lane finds its edge by binary search over the window's prefix
// offsets in shared memory, interpolates the edge in (q, t), runs forward
// kinematics once and tests every robot sphere against every obstacle sphere,
// whose positions at the lane's time are held in registers in chunks of MO
// obstacles. Robot spheres and obstacle trajectories are staged into shared
// memory by a single TMA bulk copy per CTA. FP32 CUDA-core arithmetic (no tensor
// cores: the pair tests are not a contraction).
//
// Algorithmic work per check point: S*M pair tests (8 flops each: 3 sub,
// 1 mul, 2 fma) + S sphere transforms + FK (d joint steps) + M interpolations.
//
// Verdict-only pair test. With positions taken relative to a reference point
// (the arm base, or the centre of a point robot's box), a robot sphere (c, r_s)
// and an obstacle (o, r_o) collide iff |c - o|^2 - (r_s + r_o)^2 < 0, i.e.
//   B_o + (-2 o).c + (-2 r_o) r_s  <  r_s^2 - |c|^2,   B_o = |o|^2 - r_o^2,
// which is four FMAs per pair against per-obstacle terms computed once per
// check point, plus one min per pair. In FP32 two pairs share each packed FMA
// (fma.rn.f32x2) and one three-input min; when all obstacles have one radius
// the r_s r_o term joins the per-sphere threshold and a pair costs three FMAs.
// Positions are O(1 m) relative to the reference, so the FP32 cancellation
// error near contact is about 1e-6 m; clearances keep the direct form
// |c - o| - r_s - r_o.
#pragma once

#include "stp_internal.cuh"

namespace stp {

// Per-check-point obstacle terms for the expanded pair test.
template <typename R, int MO>
struct ObsTerms {
    R ox[MO], oy[MO], oz[MO], ro[MO], B[MO];
};

template <typename R>
__device__ __forceinline__ R rmin(R a, R b) { return a < b ? a : b; }

// Packed FP32x2 helpers (Blackwell fma.rn.f32x2: two FP32 FMAs per
// instruction, each rounded once like the scalar FMA).
__device__ __forceinline__ unsigned long long pk2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void upk2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b,
                                                    unsigned long long c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

template <typename R, int MO>
__device__ __forceinline__ bool sphere_hits(R cx, R cy, R cz, R rs, const ObsTerms<R, MO>& O) {
    const R negA = rs * rs - (cx * cx + cy * cy + cz * cz);
    R m0 = rinf<R>(), m1 = rinf<R>();
#pragma unroll
    for (int j = 0; j < MO; j += 2) {
        R a = O.B[j];
        a = cx * O.ox[j] + a;
        a = cy * O.oy[j] + a;
        a = cz * O.oz[j] + a;
        a = rs * O.ro[j] + a;
        m0 = rmin(m0, a);
        if (j + 1 < MO) {
            R b = O.B[j + 1];
            b = cx * O.ox[j + 1] + b;
            b = cy * O.oy[j + 1] + b;
            b = cz * O.oz[j + 1] + b;
            b = rs * O.ro[j + 1] + b;
            m1 = rmin(m1, b);
        }
    }
    return rmin(m0, m1) < negA;
}

// Where an expression has two ways to be contracted it is written out, so that
// every kernel rounds alike.
__device__ __forceinline__ float fma_r(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_r(double a, double b, double c) { return __fma_rn(a, b, c); }
// x^2 + y^2 + z^2.
template <typename R>
__device__ __forceinline__ R norm2(R x, R y, R z) { return fma_r(z, z, fma_r(x, x, y * y)); }

// One sphere against MO obstacles by the direct form (clearances).
template <typename R, int MO>
__device__ __forceinline__ void sphere_clearance(R cx, R cy, R cz, R rs, const R (&ox)[MO], const R (&oy)[MO],
                                                 const R (&oz)[MO], const R (&orr)[MO], bool& hit, R& clr) {
#pragma unroll
    for (int j = 0; j < MO; ++j) {
        const R d2 = norm2(cx - ox[j], cy - oy[j], cz - oz[j]);
        const R rr = rs + orr[j];
        const R cl = rsqrt_r(d2) - rr;
        clr = cl < clr ? cl : clr;
        hit = hit || (d2 < rr * rr);
    }
}

// Check point of a clearance, MO obstacles at a time.
template <typename R, bool ARM, int MO>
__device__ __forceinline__ void check_point_clearance(const Geom<R>& G, const R* sm, const R (&q)[kMaxDof], R t,
                                                      bool& hit, R& clr, unsigned& pairs) {
    const R* sph = sm;
    const R* way = sm + G.off_way;
    const R* vel = sm + G.off_vel;
    const R* rad = sm + G.off_rad;
    for (int m0 = 0; m0 < G.M; m0 += MO) {
        R ox[MO], oy[MO], oz[MO], orr[MO];
#pragma unroll
        for (int j = 0; j < MO; ++j) {
            const int m = m0 + j;
            if (m < G.M) {
                obstacle_at(way + 4 * G.K * m, vel + 4 * G.K * m, G.K, t, ox[j], oy[j], oz[j]);
                orr[j] = rad[m];
            } else {
                ox[j] = oy[j] = oz[j] = R(1e18);
                orr[j] = R(0);
            }
        }
        const unsigned real = (unsigned)min(MO, G.M - m0);
        if (!ARM) {
            const R px = q[0], py = q[1], pz = (G.dof > 2) ? q[2] : R(0);
            pairs += real * (unsigned)G.S;
            for (int s = 0; s < G.S; ++s)
                sphere_clearance<R, MO>(px + sph[4 * s], py + sph[4 * s + 1], pz + sph[4 * s + 2], sph[4 * s + 3], ox,
                                        oy, oz, orr, hit, clr);
        } else {
            Frame<R> F;
            frame_identity(F);
            for (int j = 0; j <= G.dof; ++j) {
                if (j > 0) frame_step(F, G.a[j - 1], G.d[j - 1], G.ca[j - 1], G.sa[j - 1], q[j - 1] + G.th0[j - 1]);
                for (int s = G.link_start[j]; s < G.link_start[j + 1]; ++s) {
                    const R px = sph[4 * s], py = sph[4 * s + 1], pz = sph[4 * s + 2];
                    const R cx = F.o[0] + px * F.X[0] + py * F.Y[0] + pz * F.Z[0];
                    const R cy = F.o[1] + px * F.X[1] + py * F.Y[1] + pz * F.Z[1];
                    const R cz = F.o[2] + px * F.X[2] + py * F.Y[2] + pz * F.Z[2];
                    sphere_clearance<R, MO>(cx, cy, cz, sph[4 * s + 3], ox, oy, oz, orr, hit, clr);
                }
                pairs += real * (unsigned)(G.link_start[j + 1] - G.link_start[j]);
            }
        }
    }
}

// Check point in the working precision (FP64; FP32 below).
template <typename R, bool ARM, int MO>
__device__ __forceinline__ void check_point_fast(const Geom<R>& G, const R* sm, const R (&q)[kMaxDof], R t,
                                                 bool& hit, unsigned& pairs) {
    const R* sph = sm;
    const R* way = sm + G.off_way;
    const R* vel = sm + G.off_vel;
    const R* rad = sm + G.off_rad;
    for (int m0 = 0; m0 < G.M; m0 += MO) {
        ObsTerms<R, MO> O;
#pragma unroll
        for (int j = 0; j < MO; ++j) {
            const int m = m0 + j;
            if (m < G.M) {
                R x, y, z;
                obstacle_at(way + 4 * G.K * m, vel + 4 * G.K * m, G.K, t, x, y, z);
                x -= G.ref[0];
                y -= G.ref[1];
                z -= G.ref[2];
                const R r = rad[m];
                O.ox[j] = R(-2) * x;
                O.oy[j] = R(-2) * y;
                O.oz[j] = R(-2) * z;
                O.ro[j] = R(-2) * r;
                O.B[j] = x * x + y * y + z * z - r * r;
            } else {
                O.ox[j] = O.oy[j] = O.oz[j] = O.ro[j] = R(0);
                O.B[j] = R(1e30);
            }
        }
        const unsigned real = (unsigned)min(MO, G.M - m0);
        if (!ARM) {
            const R px = q[0] - G.ref[0], py = q[1] - G.ref[1], pz = ((G.dof > 2) ? q[2] : R(0)) - G.ref[2];
            for (int s = 0; s < G.S; ++s) {
                if (sphere_hits<R, MO>(px + sph[4 * s], py + sph[4 * s + 1], pz + sph[4 * s + 2], sph[4 * s + 3], O))
                    hit = true;
            }
            pairs += real * (unsigned)G.S;
        } else {
            Frame<R> F;
            frame_identity(F);
            for (int j = 0; j <= G.dof; ++j) {
                if (j > 0) frame_step(F, G.a[j - 1], G.d[j - 1], G.ca[j - 1], G.sa[j - 1], q[j - 1] + G.th0[j - 1]);
                const R ox = F.o[0] - G.ref[0], oy = F.o[1] - G.ref[1], oz = F.o[2] - G.ref[2];
                for (int s = G.link_start[j]; s < G.link_start[j + 1]; ++s) {
                    const R px = sph[4 * s], py = sph[4 * s + 1], pz = sph[4 * s + 2];
                    const R cx = ox + px * F.X[0] + py * F.Y[0] + pz * F.Z[0];
                    const R cy = oy + px * F.X[1] + py * F.Y[1] + pz * F.Z[1];
                    const R cz = oz + px * F.X[2] + py * F.Y[2] + pz * F.Z[2];
                    if (sphere_hits<R, MO>(cx, cy, cz, sph[4 * s + 3], O)) hit = true;
                }
                pairs += real * (unsigned)(G.link_start[j + 1] - G.link_start[j]);
            }
        }
    }
}

// FP32 verdict path. Obstacle position at time t from the shared-memory
// tables: the segment index is the number of waypoint times t_1..t_{K-1} not
// after max(t, t_0) (times are strictly increasing; the table is +inf padded),
// then one waypoint and one velocity record are read as float4.
__device__ __forceinline__ void obstacle_at_f32(const float4* way, const float4* vel, const float4* tim, int K,
                                                float t, float& x, float& y, float& z) {
    const float tc = fmaxf(t, way[0].x);
    const float4 ta = tim[0];
    int k = (ta.x <= tc) + (ta.y <= tc) + (ta.z <= tc) + (ta.w <= tc);
    if (K > 5) {
        const float4 tb = tim[1];
        k += (tb.x <= tc) + (tb.y <= tc) + (tb.z <= tc) + (tb.w <= tc);
    }
    const float4 w = way[k];
    const float4 v = vel[k];
    const float dtk = tc - w.x;
    x = fmaf(dtk, v.x, w.y);
    y = fmaf(dtk, v.y, w.z);
    z = fmaf(dtk, v.z, w.w);
}

__device__ __forceinline__ float min3f(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Packed obstacle terms of one chunk: lanes (2h, 2h+1) of obstacle pairs.
template <int MO>
struct ObsPacked {
    unsigned long long ox[MO / 2], oy[MO / 2], oz[MO / 2], ro[MO / 2], B[MO / 2];
};

// One robot sphere against a chunk: packed FMAs build
//   B_o + (-2 o).c [+ (-2 r_o) r_s]
// for two obstacles per instruction, three-input mins reduce them. With one
// obstacle radius R_o for all obstacles (UNI) the r_s r_o cross term is
// per-sphere and moves into the threshold r_s (r_s + 2 R_o) - |c|^2.
template <int MO, bool UNI>
__device__ __forceinline__ bool sphere_hits_packed(float cx, float cy, float cz, float rs, float ro_uni,
                                                   const ObsPacked<MO>& O) {
    const float thr = rs * (UNI ? rs + 2.f * ro_uni : rs) - (cx * cx + cy * cy + cz * cz);
    const unsigned long long CX = pk2(cx, cx), CY = pk2(cy, cy), CZ = pk2(cz, cz);
    const unsigned long long RS = UNI ? 0ull : pk2(rs, rs);
    float m0 = rinf<float>(), m1 = rinf<float>();
#pragma unroll
    for (int h = 0; h < MO / 2; ++h) {
        unsigned long long a = ffma2(CX, O.ox[h], O.B[h]);
        a = ffma2(CY, O.oy[h], a);
        a = ffma2(CZ, O.oz[h], a);
        if (!UNI) a = ffma2(RS, O.ro[h], a);
        float lo, hi;
        upk2(a, lo, hi);
        if (h & 1) m1 = min3f(m1, lo, hi);
        else m0 = min3f(m0, lo, hi);
    }
    return fminf(m0, m1) < thr;
}

template <bool ARM, int MO, bool UNI>
__device__ __forceinline__ void check_point_f32(const Geom<float>& G, const float* sm, const float (&q)[kMaxDof],
                                                float t, bool& hit, unsigned& pairs) {
    const float4* sph = reinterpret_cast<const float4*>(sm);
    const float4* way = reinterpret_cast<const float4*>(sm + G.off_way);
    const float4* vel = reinterpret_cast<const float4*>(sm + G.off_vel);
    const float4* tim = reinterpret_cast<const float4*>(sm + G.off_tim);
    const float* rad = sm + G.off_rad;
    const float ro_uni = G.ro_uni;
    for (int m0 = 0; m0 < G.M; m0 += MO) {
        ObsPacked<MO> O;
#pragma unroll
        for (int h = 0; h < MO / 2; ++h) {
            float x[2], y[2], z[2], r[2], b[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int m = m0 + 2 * h + u;
                if (m < G.M) {
                    obstacle_at_f32(way + G.K * m, vel + G.K * m, tim + 2 * m, G.K, t, x[u], y[u], z[u]);
                    if (!ARM) {
                        x[u] -= G.ref[0];
                        y[u] -= G.ref[1];
                        z[u] -= G.ref[2];
                    }
                    r[u] = UNI ? ro_uni : rad[m];
                    b[u] = x[u] * x[u] + y[u] * y[u] + z[u] * z[u] - r[u] * r[u];
                } else {
                    x[u] = y[u] = z[u] = r[u] = 0.f;
                    b[u] = 1e30f;
                }
            }
            O.ox[h] = pk2(-2.f * x[0], -2.f * x[1]);
            O.oy[h] = pk2(-2.f * y[0], -2.f * y[1]);
            O.oz[h] = pk2(-2.f * z[0], -2.f * z[1]);
            O.ro[h] = pk2(-2.f * r[0], -2.f * r[1]);
            O.B[h] = pk2(b[0], b[1]);
        }
        const unsigned real = (unsigned)min(MO, G.M - m0);
        if (!ARM) {
            const float px = q[0] - G.ref[0], py = q[1] - G.ref[1], pz = ((G.dof > 2) ? q[2] : 0.f) - G.ref[2];
            for (int s = 0; s < G.S; ++s) {
                const float4 sp = sph[s];
                if (sphere_hits_packed<MO, UNI>(px + sp.x, py + sp.y, pz + sp.z, sp.w, ro_uni, O)) hit = true;
            }
            pairs += real * (unsigned)G.S;
        } else {
            Frame<float> F;
            frame_identity(F);
            for (int j = 0; j <= G.dof; ++j) {
                if (j > 0) frame_step(F, G.a[j - 1], G.d[j - 1], G.ca[j - 1], G.sa[j - 1], q[j - 1] + G.th0[j - 1]);
                const float ox = F.o[0], oy = F.o[1], oz = F.o[2];
                const int s0 = G.link_start[j], s1 = G.link_start[j + 1];
                int s = s0;
                for (; s + 1 < s1; s += 2) {
                    const float4 sp = sph[s];
                    const float4 sq = sph[s + 1];
                    const float cx = ox + sp.x * F.X[0] + sp.y * F.Y[0] + sp.z * F.Z[0];
                    const float cy = oy + sp.x * F.X[1] + sp.y * F.Y[1] + sp.z * F.Z[1];
                    const float cz = oz + sp.x * F.X[2] + sp.y * F.Y[2] + sp.z * F.Z[2];
                    const float dx = ox + sq.x * F.X[0] + sq.y * F.Y[0] + sq.z * F.Z[0];
                    const float dy = oy + sq.x * F.X[1] + sq.y * F.Y[1] + sq.z * F.Z[1];
                    const float dz = oz + sq.x * F.X[2] + sq.y * F.Y[2] + sq.z * F.Z[2];
                    const bool h0 = sphere_hits_packed<MO, UNI>(cx, cy, cz, sp.w, ro_uni, O);
                    const bool h1 = sphere_hits_packed<MO, UNI>(dx, dy, dz, sq.w, ro_uni, O);
                    hit = hit | h0 | h1;
                }
                if (s < s1) {
                    const float4 sp = sph[s];
                    const float cx = ox + sp.x * F.X[0] + sp.y * F.Y[0] + sp.z * F.Z[0];
                    const float cy = oy + sp.x * F.X[1] + sp.y * F.Y[1] + sp.z * F.Z[1];
                    const float cz = oz + sp.x * F.X[2] + sp.y * F.Y[2] + sp.z * F.Z[2];
                    hit = hit | sphere_hits_packed<MO, UNI>(cx, cy, cz, sp.w, ro_uni, O);
                }
                pairs += real * (unsigned)(s1 - s0);
            }
        }
    }
}

template <typename R, bool ARM, int MO, bool CLEAR>
__device__ __forceinline__ void check_point(const Geom<R>& G, const R* sm, const R (&q)[kMaxDof], R t, bool& hit,
                                            R& clr, unsigned& pairs) {
    if constexpr (CLEAR) {
        check_point_clearance<R, ARM, MO>(G, sm, q, t, hit, clr, pairs);
    } else if constexpr (sizeof(R) == 4 && MO % 2 == 0) {
        if (G.uniform_ro) check_point_f32<ARM, MO, true>(G, sm, q, t, hit, pairs);
        else check_point_f32<ARM, MO, false>(G, sm, q, t, hit, pairs);
    } else {
        check_point_fast<R, ARM, MO>(G, sm, q, t, hit, pairs);
    }
}

// Self-collision of an arm state (optional): FK into a lane-private table of
// sphere centres, then the sphere predicate on the problem's pair list (pairs
// on frames at least two apart that do not touch at q = 0), read from the
// geometry blob in shared memory as a * 64 + b.
template <typename R, bool CLEAR>
__device__ __noinline__ void self_check(const Geom<R>& G, const R* sm, const R (&q)[kMaxDof], bool& hit, R& clr) {
    R c[kMaxSpheres][3];
    const R* sph = sm;
    Frame<R> F;
    frame_identity(F);
    for (int j = 0; j <= G.dof; ++j) {
        if (j > 0) frame_step(F, G.a[j - 1], G.d[j - 1], G.ca[j - 1], G.sa[j - 1], q[j - 1] + G.th0[j - 1]);
        for (int s = G.link_start[j]; s < G.link_start[j + 1]; ++s) {
            const R px = sph[4 * s], py = sph[4 * s + 1], pz = sph[4 * s + 2];
            for (int i = 0; i < 3; ++i) c[s][i] = F.o[i] + px * F.X[i] + py * F.Y[i] + pz * F.Z[i];
        }
    }
    const R* pairs = sm + G.off_self;
    for (int k = 0; k < G.n_self; ++k) {
        const int code = (int)pairs[k];
        const int a = code >> 6, b = code & 63;
        const R dx = c[a][0] - c[b][0], dy = c[a][1] - c[b][1], dz = c[a][2] - c[b][2];
        const R d2 = norm2(dx, dy, dz);
        const R rr = sph[4 * a + 3] + sph[4 * b + 3];
        if (d2 < rr * rr) {
            hit = true;
            if (!CLEAR) return;
        }
        if (CLEAR) {
            const R cl = rsqrt_r(d2) - rr;
            clr = cl < clr ? cl : clr;
        }
    }
}

template <typename R>
__device__ __forceinline__ void atomic_min_r(R* addr, R v);
template <>
__device__ __forceinline__ void atomic_min_r<float>(float* addr, float v) {
    atomicMin(reinterpret_cast<int*>(addr), ord_enc(v));
}
template <>
__device__ __forceinline__ void atomic_min_r<double>(double* addr, double v) {
    atomicMin(reinterpret_cast<long long*>(addr), ord_enc(v));
}

// Most edges per shared-memory window.
constexpr int kWin = 64;

// smem_raw: the geometry blob (staged by one TMA bulk copy) and the window's
// offsets. A CTA's share of the edges is cut into up to four even windows of at
// most kWin edges, so that CTAs with harder edges take fewer of them: no more
// windows than there are lanes to fill with check points (by the batch's mean; a
// window costs three barriers and an atomic), and none that a few CTAs take alone
// at the end. 65,536 seven-axis edges: 2.77 ms with five windows to some CTAs,
// 2.57 ms with windows of kWin, 2.48 ms so.
template <typename R, bool ARM, int MO, bool CLEAR>
__device__ __forceinline__ void validate_full_body(const Geom<R>& G, const EdgeBatch<R>& E, unsigned char* smem_raw) {
    __shared__ __align__(8) uint64_t bar;
    __shared__ int s_win, s_size;  // window number, edges per window
    R* sm = reinterpret_cast<R*>(smem_raw);
    const int n = E.n_host;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_expect_tx(&bar, G.blob_bytes);
        bulk_g2s(sm, G.blob, G.blob_bytes, &bar);
        const int grid = gridDim.x;
        // Edges that fill the lanes, by the batch's mean; windows to a CTA.
        const int fill = max(1, (int)fminf((float)kWin, (float)blockDim.x * (float)n / fmaxf((float)E.off[n], 1.f)));
        const int cuts = min(4, (n + fill * grid - 1) / (fill * grid));
        s_size = min(kWin, (n + cuts * grid - 1) / (cuts * grid));
    }
    __syncthreads();
    if (!mbar_wait(&bar, 0)) {
        if (threadIdx.x == 0 && E.err) atomicOr(E.err, kErrTimeout);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    unsigned long long done = 0, pairs_total = 0;

    // One check point g of edge e: interpolate, run FK and the pair tests.
    auto process = [&](long long g, int e, long long e_off) {
        const int c = E.cnt[e];
        const int jj = (int)(g - e_off) + 1;
        const R s = R(jj) / R(c);
        const R* qa = E.qa + (size_t)e * E.qstride;
        const R* qb = E.qb + (size_t)e * E.qstride;
        R q[kMaxDof];
        bool hit = false;
#pragma unroll
        for (int i = 0; i < kMaxDof; ++i) {
            if (i < G.dof) {
                q[i] = qa[i] + s * (qb[i] - qa[i]);
                hit = hit || (q[i] < G.qlo[i]) || (q[i] > G.qhi[i]);
            } else {
                q[i] = R(0);
            }
        }
        const R ta = E.ta[e];
        const R t = ta + s * (E.tb[e] - ta);
        R clr = rinf<R>();
        unsigned pairs = 0;
        check_point<R, ARM, MO, CLEAR>(G, sm, q, t, hit, clr, pairs);
        if (ARM && G.n_self > 0 && (CLEAR || !hit)) self_check<R, CLEAR>(G, sm, q, hit, clr);
        if (hit) E.hit[e] = 1;
        if (CLEAR) atomic_min_r<R>(E.clear + e, clr);  // order-encoded, decoded by launch_finish_batch
        ++done;
        pairs_total += pairs;
    };

    // CTAs take windows of consecutive edges from the work counter as they
    // finish the previous one (the batch ends within one window of balance),
    // stage the window's offsets and spread its check points over their warps.
    long long* woff = reinterpret_cast<long long*>(smem_raw + G.blob_bytes);
    for (;;) {
        __syncthreads();   // the previous window's offsets are no longer read
        if (threadIdx.x == 0) s_win = atomicAdd(E.next, 1);
        __syncthreads();
        const int win = s_size, w0 = s_win * win;
        if (w0 >= n) break;
        const int wn = min(win, n - w0);
        for (int i = threadIdx.x; i <= wn; i += blockDim.x) woff[i] = E.off[w0 + i];
        __syncthreads();
        const long long ob = woff[0], oe = woff[wn];
        for (long long g = ob + warp * 32 + lane; g < oe; g += wpb * 32) {
            int lo = 0, hi = wn - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (woff[mid] <= g) lo = mid;
                else hi = mid - 1;
            }
            process(g, w0 + lo, woff[lo]);
        }
    }
    if (E.points_done) {
        for (int o = 16; o > 0; o >>= 1) done += __shfl_xor_sync(0xffffffffu, done, o);
        if (lane == 0 && done) atomicAdd(E.points_done, done);
    }
    if (E.pairs_done) {
        for (int o = 16; o > 0; o >>= 1) pairs_total += __shfl_xor_sync(0xffffffffu, pairs_total, o);
        if (lane == 0 && pairs_total) atomicAdd(E.pairs_done, pairs_total);
    }
}

}  // namespace stp
