// Edge validation by bounded motion (verdicts and clearances of space-time
// edges against moving obstacles), shared by the stand-alone edge batch, the
// planner's per-step and batched launches and the persistent planner kernel.
//
// An edge's verdict is the OR over its check points j = 1..c of "collides",
// its clearance the minimum over them. Between neighbouring check points a
// sphere on frame f and an obstacle cannot approach by more than
//   delta_f = (sum_{j < f} |dq_j| R_jf + v_obs |dt|) / c,
// with R_jf the largest distance of a sphere of frame f from the axis of joint
// j and v_obs the largest obstacle speed (fixed per problem, on the host). A
// point whose spheres have clearances d_s therefore decides its neighbours too:
// every check point within min_s floor((d_s - mu) / delta_f(s)) of it is free
// (or, for the clearance, above the smallest one found so far). mu covers the
// rounding of every quantity involved, several times over, so a skipped point
// is one whose own arithmetic would have said "free": verdicts and clearances
// are those of checking every point, bit for bit. The points are visited by
// bisection: a stack holds the undecided index intervals of an edge; the middle
// of an interval is evaluated and what it does not decide is pushed back as
// at most two intervals. On random 0.5 rad steps of the six-axis arm (50 check
// points, 61 % colliding) this evaluates 3.4 points an edge (6.4 with one bound
// for the whole arm), on planner bridges (hundreds of points) 2-10.
//
// Where the bound does not apply every point is evaluated: the stretch of an
// edge on or outside the configuration box (the box test is per point),
// self-collision pairs (their relative motion is not bounded here), non-finite
// inputs, and geometry too large for the rounding margins (lip_ok = 0).
//
// Arms evaluate a point in two passes. The near pass works in FP32 on the
// expanded pair test of stp_validate_body.cuh (the same operations in the same
// order for every pair) and yields the bound; in an FP32 verdict its sign is
// the result. Clearances, and FP64 problems, take the exact pass as well, in
// their own precision, where the near pass leaves the answer open: a clearance
// only where the point may be lower than the smallest so far, an FP64 verdict
// only where the FP32 distance is within mu of contact (about one point in a
// thousand; the FP64 units run at 1/64 of the FP32 rate).
//
// Mapping: L lanes share a check point, so a warp evaluates 32 / L. Nothing is
// computed twice: lane r interpolates joint r and its sine and cosine, lanes 0-2
// carry one row each of the link frames (rows are independent), lane r
// interpolates obstacle pair r and lane r tests spheres r, r + L, ... against
// all obstacles; frames and obstacle terms pass through the warp's own shared
// memory. A point is a chain of about 600 instructions (L = 8) instead of the
// 3,200 of one lane per point.
//
// Two bodies share that evaluation. edge_pool: a CTA takes a few edges and
// evaluates all their undecided intervals together, level by level (a block
// barrier between levels), so the few edges that need many points spread over
// every warp instead of holding one; for the planner's batches, others of up to
// about 100,000 edges (FP64 34,000, point robots 15,000) and, at any size, those
// without a bound. edge_stream: each lane group takes an edge of its own from the
// stream and needs no barrier; for large batches, with L = 4 in FP32 (less of the
// chain is spent on the joints). Which points of an edge are evaluated for a
// verdict depends on the edge and the launch alone, not on timing, so the work
// counters repeat from run to run.
//
// Measured on one GB300, against one lane per check point over every point:
// 2^20 UR5e edges 6.0 -> 0.92 ms, 61 of them 107 -> 17 us a call, clearances of
// 9,973 seven-axis edges among 64 obstacles 2.59 -> 0.90 ms, 2,003 of them in
// FP64 13.0 -> 0.14 ms. The stream issues on 41 % of its cycles with 2.6 of 6
// stall cycles an instruction on shared memory and shuffles: what bounds it is
// the latency of a point's chain at the 16-24 warps an SM that registers and
// scratch allow.
#pragma once

#include "stp_validate_body.cuh"

namespace stp {

constexpr int kPoolLanes = 8;    // lanes per check point in edge_pool (and of FP64 and clearance streams)
constexpr int kStreamLanes = 4;  // in edge_stream (FP32 verdicts, point robots)
constexpr int kEdgeStack = 20;   // edge_stream: intervals per group (beyond: one point at a time)
constexpr int kHeld = 11;        // edge_stream: per edge held, eight bounds, margin, first and last covering point
constexpr int kPoolSlots = 16;   // edge_pool: edges of a CTA at a time
constexpr int kPoolList = 512;   // and undecided intervals (beyond half of it: one point at a time)
constexpr int kFrameStride = 8 * 12 + 4;  // R values per point: 8 frames x 3 rows x (X, Y, Z, o), padded
static_assert(kMaxDof < 8, "frames 0..7 in eight slots");

// Obstacles whose terms are held in shared memory at a time: 64, or 32 when a
// warp evaluates eight points.
__host__ __device__ inline int edge_chunk_of(int M, int L) {
    const int most = L >= 8 ? 64 : 32, m = (M + 15) / 16 * 16;
    return m < most ? (m > 0 ? m : 16) : most;
}
// Obstacle terms of one point (a pair: -2x, -2y, -2z, B, then -2 r_o of every
// pair), padded so that the points start on different banks.
__host__ __device__ inline int edge_obs_stride(int chunk) { return chunk * 5 + 4; }
__host__ __device__ inline int edge_self_stride(int S) { return (3 * S + 3) / 4 * 4; }

// Shared memory of one warp with 32 / L points, in this order. edge_stream: the
// groups' intervals, steps per metre by frame of each group's edge, the same
// with margin and range for the 32 edges a warp holds. Both, for arms: the near
// pass's frames and obstacle terms (and sphere centres for self-collision), and
// in clearances and FP64 (exact) a distance per sphere and the exact pass's
// frames (and centres).
struct EdgeShared {
    int steps, held, near, dist, exact, bytes;  // byte offsets in a warp's part, and its size
};
template <typename R>
__host__ __device__ inline EdgeShared edge_shared(int arm, int S, int M, int n_self, int L, bool pool, bool exact) {
    const int NP = 32 / L;
    EdgeShared e;
    e.steps = pool ? 0 : NP * kEdgeStack * 8;
    e.held = pool ? 0 : e.steps + NP * 8 * 4;
    e.near = pool ? 0 : e.held + 32 * kHeld * 4;
    int b = e.near;
    if (arm) {
        b += NP * (kFrameStride + edge_obs_stride(edge_chunk_of(M, L))) * 4;
        if (n_self > 0 && !exact) b += NP * edge_self_stride(S) * 4;
    }
    e.dist = b;
    if (arm && exact) b += NP * kMaxSpheres * 4;
    e.exact = b;
    if (arm && exact) {
        if (sizeof(R) == 8) b += NP * kFrameStride * (int)sizeof(R);
        if (n_self > 0) b += NP * edge_self_stride(S) * (int)sizeof(R);
    }
    e.bytes = (b + 15) / 16 * 16;
    return e;
}
// edge_pool's edges and interval lists (after the tables).
template <typename R>
struct PoolShared {
    R q[kPoolSlots][16];  // q_a (8), q_b (8)
    R t[kPoolSlots][2];
    R best[kPoolSlots];   // clearances: order-encoded smallest distance so far
    float dv[kPoolSlots][8];
    float mu[kPoolSlots];
    int c[kPoolSlots], edge[kPoolSlots];
    int hit[kPoolSlots];  // level at which a collision was found (0: none)
    int2 iv[2][kPoolList];
    unsigned char slot[2][kPoolList];
    int n[3], nslot;
    long long base;
};
template <typename R>
__host__ __device__ constexpr int pool_bytes() { return ((int)sizeof(PoolShared<R>) + 15) / 16 * 16; }
// Edges a CTA takes at a time and the intervals an edge starts with: as many as
// keep the CTA's lane groups busy in the first level.
__host__ __device__ inline int pool_edges(int n, int ncta) {
    const int b = (n + ncta - 1) / ncta;
    return b < 1 ? 1 : (b > kPoolSlots ? kPoolSlots : b);
}
__host__ __device__ inline int pool_pieces(int edges) { return edges <= 1 ? 16 : (edges <= 8 ? 8 : 4); }

// Block-wide tables after the blob: per joint th0, q_lo, q_hi; reach [7][8];
// the frame of each sphere.
template <typename R>
__host__ __device__ constexpr int edge_table_bytes() {
    return 4 * 8 * (int)sizeof(R) + 8 * 8 * 4 + kMaxSpheres * 4;
}

// Points x < j <= y of an edge lie inside the configuration box by more than the
// rounding of their joint values, so a point among them may decide others there.
// An edge's first intervals end at x and y; those outside, where every point is
// evaluated, hold minus their last point, and so do the parts of them.
// s1, s2: where the edge enters and leaves that inner box (of c check points).
__device__ __forceinline__ int2 box_range(float s1, float s2, int c) {
    const int x = s1 > 0.f ? (int)((s1 + 1e-5f) * (float)c) : 0;
    const int y = s2 < 1.f ? (int)((s2 - 1e-5f) * (float)c) : c;
    return x < y ? make_int2(x, y) : make_int2(0, 0);
}
// A joint value between qa and qb is rounded by less than this (qm: |qa| + |qb|).
__device__ __forceinline__ float box_margin(float qm) { return 4e-6f * (1.f + qm); }
// One side of one joint: a and b, the distances from it beyond the margin at the ends.
__device__ __forceinline__ void box_side(float a, float b, float& s1, float& s2) {
    if (a > 0.f && b > 0.f) return;
    const float x = a / (a - b);  // the crossing
    if (!(x >= 0.f && x <= 1.f) || !(a > 0.f || b > 0.f)) s2 = -1.f;  // outside throughout, or not a number
    else if (a > 0.f) s2 = fminf(s2, x);
    else s1 = fmaxf(s1, x);
}
template <typename R>
__device__ __forceinline__ void box_joint(R qa, R qb, R lo, R hi, float& s1, float& s2) {
    const float bt = box_margin(fabsf((float)qa) + fabsf((float)qb));
    box_side((float)(qa - lo) - bt, (float)(qb - lo) - bt, s1, s2);
    box_side((float)(hi - qa) - bt, (float)(hi - qb) - bt, s1, s2);
}

__device__ __forceinline__ float floor_steps(float x) { return x > 0.f ? fminf(x, 1e9f) : 0.f; }  // NaN: 0
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// Check points of an edge in double, as defined for stp_check_edges; FP32
// inputs decide in FP32 whenever the quotient is not within its rounding (a few
// 1e-6 relative) of an integer, which saves the double square root and
// division (the FP64 units are 1/64 of the FP32 ones).
template <typename R>
__device__ __forceinline__ int edge_count(const R (&qa)[kMaxDof], const R (&qb)[kMaxDof], R ta, R tb, int dof,
                                          double vmax, double res) {
    if constexpr (sizeof(R) == 4) {
        float s2 = 0.f;
#pragma unroll
        for (int i = 0; i < kMaxDof; ++i)
            if (i < dof) {
                const float d = qb[i] - qa[i];
                s2 = fmaf(d, d, s2);
            }
        const float x = fmaxf(sqrtf(s2), (float)vmax * fabsf(tb - ta)) / (float)res - 1e-3f;
        const float f = floorf(x), tol = 4e-6f * x + 4e-6f;
        if (x > 0.f && x < 1e5f && x - f > tol && x - f < 1.f - tol) return (int)f + 1;
    }
    double s2 = 0.0;
#pragma unroll
    for (int i = 0; i < kMaxDof; ++i)
        if (i < dof) {
            const double dd = (double)qb[i] - (double)qa[i];
            s2 = __dadd_rn(s2, __dmul_rn(dd, dd));
        }
    const double Lg = fmax(sqrt(s2), __dmul_rn(vmax, fabs((double)tb - (double)ta)));
    const double c = ceil(Lg / res - 1e-3);
    return c < 1.0 ? 1 : (int)c;
}

// KS spheres per lane against the obstacle pairs in shared memory (FP32): e of
// each sphere, the smallest d^2 - (r_s + r_o)^2.
template <int KS, bool UNI>
__device__ __forceinline__ void pairs_f32(const float (&cx)[KS], const float (&cy)[KS], const float (&cz)[KS],
                                           const float (&rs)[KS], float ro_uni, const float* ob, const float* ro,
                                           int np, float (&e)[KS]) {
    unsigned long long CX[KS], CY[KS], CZ[KS], RS[KS];
    float m[KS], thr[KS];
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        thr[k] = rs[k] * (UNI ? rs[k] + 2.f * ro_uni : rs[k]) - (cx[k] * cx[k] + cy[k] * cy[k] + cz[k] * cz[k]);
        CX[k] = pk2(cx[k], cx[k]);
        CY[k] = pk2(cy[k], cy[k]);
        CZ[k] = pk2(cz[k], cz[k]);
        RS[k] = UNI ? 0ull : pk2(rs[k], rs[k]);
        m[k] = rinf<float>();
    }
#pragma unroll 4
    for (int h = 0; h < np; ++h) {
        const ulonglong2 a = reinterpret_cast<const ulonglong2*>(ob)[2 * h];
        const ulonglong2 b = reinterpret_cast<const ulonglong2*>(ob)[2 * h + 1];
        unsigned long long r = 0;
        if (!UNI) r = reinterpret_cast<const unsigned long long*>(ro)[h];
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            unsigned long long v = ffma2(CX[k], a.x, b.y);
            v = ffma2(CY[k], a.y, v);
            v = ffma2(CZ[k], b.x, v);
            if (!UNI) v = ffma2(RS[k], r, v);
            float lo, hi;
            upk2(v, lo, hi);
            m[k] = min3f(m[k], lo, hi);
        }
    }
#pragma unroll
    for (int k = 0; k < KS; ++k) e[k] = m[k] - thr[k];
}

// Obstacle m at time t: position relative to the pair tests' reference point
// (verdicts) or absolute (clearances), and radius.
template <typename R, bool ARM, bool CLEAR>
__device__ __forceinline__ void obstacle_terms(const Geom<R>& G, const R* sm, int m, R t, R& x, R& y, R& z, R& ro) {
    const R* way = sm + G.off_way;
    const R* vel = sm + G.off_vel;
    if constexpr (sizeof(R) == 4 && !CLEAR) {
        obstacle_at_f32(reinterpret_cast<const float4*>(way) + G.K * m, reinterpret_cast<const float4*>(vel) + G.K * m,
                        reinterpret_cast<const float4*>(sm + G.off_tim) + 2 * m, G.K, t, x, y, z);
        ro = G.uniform_ro ? G.ro_uni : sm[G.off_rad + m];
    } else {
        obstacle_at(way + 4 * G.K * m, vel + 4 * G.K * m, G.K, t, x, y, z);
        ro = sm[G.off_rad + m];
    }
    if (!CLEAR && (!ARM || sizeof(R) == 8)) {
        x -= G.ref[0];
        y -= G.ref[1];
        z -= G.ref[2];
    }
}

// Centre and radius of sphere s at the frames fr.
template <typename R>
__device__ __forceinline__ void sphere_centre(const R* sph, const R* F, int s, R& cx, R& cy, R& cz, R& rs) {
    if constexpr (sizeof(R) == 4) {
        const float4 v = reinterpret_cast<const float4*>(sph)[s];
        const float4 f0 = reinterpret_cast<const float4*>(F)[0], f1 = reinterpret_cast<const float4*>(F)[1],
                     f2 = reinterpret_cast<const float4*>(F)[2];
        rs = v.w;
        cx = f0.w + v.x * f0.x + v.y * f0.y + v.z * f0.z;
        cy = f1.w + v.x * f1.x + v.y * f1.y + v.z * f1.z;
        cz = f2.w + v.x * f2.x + v.y * f2.y + v.z * f2.z;
    } else {
        const R px = sph[4 * s], py = sph[4 * s + 1], pz = sph[4 * s + 2];
        rs = sph[4 * s + 3];
        cx = F[3] + px * F[0] + py * F[1] + pz * F[2];
        cy = F[7] + px * F[4] + py * F[5] + pz * F[6];
        cz = F[11] + px * F[8] + py * F[9] + pz * F[10];
    }
}

// Near-pass scratch of a group.
struct PointScratch {
    float* fr;  // frames [8][3][4]
    float* ob;  // obstacle terms
    float* ro;  // -2 r_o
    float* sc;  // sphere centres (self-collision) or nullptr
    int chunk;
};

// Frames of the arm at the group's joint angles (joint j at lane j % L).
template <typename R, int L>
__device__ __forceinline__ void arm_frames(const Geom<R>& G, R* fr, int r, const R (&theta)[8 / L]) {
    R sn[8 / L], cs[8 / L];
#pragma unroll
    for (int i = 0; i < 8 / L; ++i) sincos_r(theta[i], &sn[i], &cs[i]);
    // Lane i < 3 carries row i of the frames (columns X, Y, Z and origin o).
    R X = r == 0 ? R(1) : R(0), Y = r == 1 ? R(1) : R(0), Z = r == 2 ? R(1) : R(0), o = R(0);
    auto put = [&](int j) {
        if (r < 3) {
            R* p = fr + 12 * j + 4 * r;
            if constexpr (sizeof(R) == 4) {
                *reinterpret_cast<float4*>(p) = make_float4(X, Y, Z, o);
            } else {
                reinterpret_cast<double2*>(p)[0] = make_double2(X, Y);
                reinterpret_cast<double2*>(p)[1] = make_double2(Z, o);
            }
        }
    };
    put(0);
#pragma unroll
    for (int j = 0; j < kMaxDof; ++j) {
        if (j < G.dof) {
            const R s = __shfl_sync(0xffffffffu, sn[j / L], j % L, L), c = __shfl_sync(0xffffffffu, cs[j / L], j % L, L);
            const R u = fma_r(c, X, s * Y);
            const R w = fma_r(c, Y, -(s * X));
            const R z = Z;
            X = u;
            Y = fma_r(G.sa[j], z, G.ca[j] * w);
            Z = fma_r(G.ca[j], z, -(G.sa[j] * w));
            o = fma_r(G.d[j], z, fma_r(G.a[j], u, o));
            put(j + 1);
        }
    }
}

// Terms of obstacles m0 .. m0 + mc - 1 at time t (a pair per lane and round).
template <int L>
__device__ __forceinline__ void obstacle_chunk(const Geom<float>& G, const float* sm, const PointScratch& P, int r,
                                               int m0, int mc, float t) {
    for (int h = r; 2 * h < mc; h += L) {
        float x[2], y[2], z[2], rr[2], b[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (2 * h + u < mc) {
                obstacle_terms<float, true, false>(G, sm, m0 + 2 * h + u, t, x[u], y[u], z[u], rr[u]);
                b[u] = x[u] * x[u] + y[u] * y[u] + z[u] * z[u] - rr[u] * rr[u];
            } else {
                x[u] = y[u] = z[u] = rr[u] = 0.f;
                b[u] = 1e30f;
            }
        }
        float* p = P.ob + 8 * h;
        reinterpret_cast<float4*>(p)[0] = make_float4(-2.f * x[0], -2.f * x[1], -2.f * y[0], -2.f * y[1]);
        reinterpret_cast<float4*>(p)[1] = make_float4(-2.f * z[0], -2.f * z[1], b[0], b[1]);
        if (!G.uniform_ro) *reinterpret_cast<float2*>(P.ro + 2 * h) = make_float2(-2.f * rr[0], -2.f * rr[1]);
    }
}

// Self-collision of the group's state (every sphere's centre in sc).
template <typename R, bool CLEAR, int L>
__device__ __forceinline__ void self_pairs(const Geom<R>& G, const R* sph, const R* pairs, const R* sc, int r, bool& hit,
                                           R& clr) {
    for (int k = r; k < G.n_self; k += L) {
        const int code = (int)pairs[k];
        const int a = code >> 6, b = code & 63;
        const R dx = sc[3 * a] - sc[3 * b], dy = sc[3 * a + 1] - sc[3 * b + 1], dz = sc[3 * a + 2] - sc[3 * b + 2];
        const R d2 = norm2(dx, dy, dz);
        const R rr = sph[4 * a + 3] + sph[4 * b + 3];
        hit = hit || d2 < rr * rr;
        if (CLEAR) {
            const R cl = rsqrt_r(d2) - rr;
            clr = cl < clr ? cl : clr;
        }
    }
}

// Lower bound of a pair's distance from e = d^2 - rr^2, less its rounding, for
// any radius sum rr between rr_min and rr_max.
__device__ __forceinline__ float distance_bound(const Geom<float>& G, float e, float rr_min, float rr_max) {
    e -= G.lip_eps;
    if (e >= 0.f) return sqrt_approx(fmaf(rr_max, rr_max, e)) - rr_max;
    const float x = fmaf(rr_min, rr_min, e);
    return x >= 0.f ? sqrt_approx(x) - rr_min : -sqrt_approx(-e);
}

// Near pass over KS spheres per lane: e, and the check points that each sphere's
// distance decides (dv: steps per metre by frame) or, with DIST, a lower bound
// of the distance by sphere (lb).
template <int KS, bool DIST, int L>
__device__ __forceinline__ void near_batch(const Geom<float>& G, const float* sm, const int* sfr, const PointScratch& P,
                                           const float* dv, int s0, int r, int m0, int mc, float rrmu, float mu,
                                           float& e, float& steps, float* lb) {
    float cx[KS], cy[KS], cz[KS], rs[KS], es[KS];
    int sf[KS];
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const int s = min(s0 + r + L * k, G.S - 1);  // beyond the last: that sphere again
        sf[k] = sfr[s];
        sphere_centre<float>(sm, P.fr + 12 * sf[k], s, cx[k], cy[k], cz[k], rs[k]);
        if (P.sc) {
            P.sc[3 * s] = cx[k];
            P.sc[3 * s + 1] = cy[k];
            P.sc[3 * s + 2] = cz[k];
        }
    }
    if constexpr (DIST) {
        // Obstacles are sorted by radius: sixteen at a time the radii span little, and
        // the bound is tight.
        float d[KS];
#pragma unroll
        for (int k = 0; k < KS; ++k) d[k] = rinf<float>();
        const int step = G.uniform_ro ? mc : 16;
        for (int o = 0; o < mc; o += step) {
            const int oc = min(step, mc - o), np = (oc + 1) >> 1;
            float lo = G.ro_uni, hi = G.ro_uni;
            if (G.uniform_ro) {
                pairs_f32<KS, true>(cx, cy, cz, rs, G.ro_uni, P.ob, P.ro, np, es);
            } else {
                pairs_f32<KS, false>(cx, cy, cz, rs, G.ro_uni, P.ob + 4 * o, P.ro + o, np, es);
                lo = sm[G.off_rad + m0 + o];
                hi = sm[G.off_rad + m0 + o + oc - 1];
            }
#pragma unroll
            for (int k = 0; k < KS; ++k) {
                e = fminf(e, es[k]);
                d[k] = fminf(d[k], distance_bound(G, es[k], (rs[k] + lo) * 0.999999f, (rs[k] + hi) * 1.000001f));
            }
        }
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const int s = s0 + r + L * k;
            if (s < G.S) {
                const float x = d[k] - mu;
                lb[s] = m0 == 0 ? x : fminf(lb[s], x);
                steps = fminf(steps, x);
            }
        }
    } else {
        const int np = (mc + 1) >> 1;
        if (G.uniform_ro) pairs_f32<KS, true>(cx, cy, cz, rs, G.ro_uni, P.ob, P.ro, np, es);
        else pairs_f32<KS, false>(cx, cy, cz, rs, G.ro_uni, P.ob, P.ro, np, es);
        const float rr2 = G.lip_rr * G.lip_rr;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            e = fminf(e, es[k]);
            steps = fminf(steps, (sqrt_approx(es[k] + rr2) - rrmu) * dv[sf[k]]);
        }
    }
}

// Near pass (FP32) of one check point per lane group: the lane's smallest
// e = d^2 - (r_s + r_o)^2 and the steps its spheres decide (DIST: the smallest
// distance bound less the margin, by sphere in lb). The warp runs it together.
template <bool DIST, int L>
__device__ __forceinline__ void near_pass(const Geom<float>& G, const float* sm, const int* sfr, const PointScratch& P,
                                          const float* dv, int r, const float (&theta)[8 / L], float t, float mu,
                                          float& e, float& steps, float* lb) {
    arm_frames<float, L>(G, P.fr, r, theta);
    const float rrmu = G.lip_rr + mu;
    int m0 = 0;
    do {
        const int mc = min(P.chunk, G.M - m0);
        if (m0 > 0) __syncwarp();  // the previous chunk's terms are no longer read
        obstacle_chunk<L>(G, sm, P, r, m0, mc, t);
        __syncwarp();
        int s0 = 0;
        for (; s0 + 2 * L < G.S; s0 += 4 * L)
            near_batch<4, DIST, L>(G, sm, sfr, P, dv, s0, r, m0, mc, rrmu, mu, e, steps, lb);
        if (s0 < G.S) near_batch<2, DIST, L>(G, sm, sfr, P, dv, s0, r, m0, mc, rrmu, mu, e, steps, lb);
        m0 += P.chunk;
    } while (m0 < G.M);
}

// Sphere s of the group's state against every obstacle, in the working
// precision (lane r: obstacles r, r + L, ...): a collision, and with CLEAR the
// smallest distance, of the group. ob, ro: the near pass's terms where they hold
// every obstacle in that precision (-2 times the positions and radii, an exact
// scaling), else nullptr.
template <typename R, bool CLEAR, int L>
__device__ __forceinline__ void exact_sphere(const Geom<R>& G, const R* blob, const R* F, const R* ob, const R* ro_,
                                             int s, int r, R t, bool& hit, R& clr) {
    R cx, cy, cz, rs;
    sphere_centre<R>(blob, F, s, cx, cy, cz, rs);
    const R negA = rs * rs - (cx * cx + cy * cy + cz * cz);
    bool h = false;
    R best = rinf<R>();
    for (int m = r; m < G.M; m += L) {
        R x, y, z, ro;
        if (CLEAR && ob) {
            const R* o = ob + 8 * (m >> 1) + (m & 1);
            x = R(-0.5) * o[0];
            y = R(-0.5) * o[2];
            z = R(-0.5) * o[4];
            ro = G.uniform_ro ? G.ro_uni : R(-0.5) * ro_[m];
        } else {
            obstacle_terms<R, true, CLEAR>(G, blob, m, t, x, y, z, ro);
        }
        if constexpr (CLEAR) {
            const R d2 = norm2(cx - x, cy - y, cz - z);
            const R rr = rs + ro;
            const R cl = rsqrt_r(d2) - rr;
            best = cl < best ? cl : best;
            h = h || (d2 < rr * rr);
        } else {
            R a = x * x + y * y + z * z - ro * ro;
            a = cx * (R(-2) * x) + a;
            a = cy * (R(-2) * y) + a;
            a = cz * (R(-2) * z) + a;
            a = rs * (R(-2) * ro) + a;
            h = h || a < negA;
        }
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
        if (CLEAR) best = rmin(best, __shfl_xor_sync(0xffffffffu, best, o));
        h = h | (bool)__shfl_xor_sync(0xffffffffu, (int)h, o);
    }
    hit = h;
    clr = best;
}

// Exact pass of one check point per lane group, in the working precision,
// over the spheres whose distance bound leaves the answer open: lb <= val
// (clearances: the smallest distance so far, verdicts: 0), or over all of them.
// open: the group takes part. hit and val are updated; the warp runs it together.
template <typename R, bool CLEAR, int L>
__device__ __noinline__ void exact_pass(const Geom<R>& G, const R* blob, const int* sfr, R* fr, const R* ob,
                                        const R* ro, R* sc, const float* lb, int r, R theta, R t, bool open, bool all, bool& hit_io, R& val_io) {
    constexpr unsigned kFull = 0xffffffffu;
    bool hit = hit_io;
    R val = val_io;
    if constexpr (sizeof(R) == 8) {
        const R th[1] = {theta};
        arm_frames<R, L>(G, fr, r, th);
    }
    __syncwarp();
    auto run = [&](int s, bool on) {
        bool h;
        R c;
        exact_sphere<R, CLEAR, L>(G, blob, fr + 12 * sfr[s], ob, ro, s, r, t, h, c);
        if (on) {
            hit = hit || h;
            if (CLEAR) val = rmin(val, c);
        }
    };
    if constexpr (CLEAR) {
        // The sphere with the lowest bound first: it leaves few others open.
        float b = rinf<float>();
        int s = 0;
        for (int k = r; k < G.S; k += L)
            if (lb[k] < b) {
                b = lb[k];
                s = k;
            }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) {
            const float b2 = __shfl_xor_sync(kFull, b, o);
            const int s2 = __shfl_xor_sync(kFull, s, o);
            if (b2 < b || (b2 == b && s2 < s)) {
                b = b2;
                s = s2;
            }
        }
        run(s, open);
    }
    for (int k0 = 0; k0 < G.S; k0 += L) {
        const float b = k0 + r < G.S ? lb[k0 + r] : rinf<float>();
        int next = 0;  // the group's spheres below k0 + next are done
        for (int it = 0; it < L; ++it) {  // each round takes a sphere of every group that has one open
            const bool cand = open && k0 + r < G.S && r >= next && (all || !(b > (float)val)) && (CLEAR || !hit);
            const unsigned m = (__ballot_sync(kFull, cand) >> ((threadIdx.x & 31) / L * L)) & ((1u << L) - 1u);
            if (!__any_sync(kFull, m != 0)) break;
            const int k = m ? __ffs(m) - 1 : 0;
            run(min(k0 + k, G.S - 1), m != 0);
            if (m) next = k + 1;
        }
    }
    if (sc) {
        for (int s = r; s < G.S; s += L) {
            R cx, cy, cz, rs;
            sphere_centre<R>(blob, fr + 12 * sfr[s], s, cx, cy, cz, rs);
            sc[3 * s] = cx;
            sc[3 * s + 1] = cy;
            sc[3 * s + 2] = cz;
        }
        __syncwarp();
        bool h = false;
        R c = rinf<R>();
        self_pairs<R, CLEAR, L>(G, blob, blob + G.off_self, sc, r, h, c);
        if (open) {
            hit = hit || h;  // of the lane
            if (CLEAR) val = rmin(val, c);
        }
    }
    hit_io = hit;
    val_io = val;
}

// Point robots (few spheres): the lane tests its obstacles against all spheres.
// val: the lane's smallest e (verdicts) or distance (clearances).
template <typename R, bool CLEAR, int L>
__device__ __forceinline__ void point_robot(const Geom<R>& G, const R* sm, int r, R q, R t, bool& hit, R& val) {
    constexpr unsigned kFull = 0xffffffffu;
    R px = __shfl_sync(kFull, q, 0, L), py = __shfl_sync(kFull, q, 1, L), pz = __shfl_sync(kFull, q, 2, L);
    if (G.dof <= 2) pz = R(0);
    if constexpr (!CLEAR) {
        px -= G.ref[0];
        py -= G.ref[1];
        pz -= G.ref[2];
    }
    for (int h = r; 2 * h < G.M; h += L) {
        R x[2], y[2], z[2], rr[2], b[2];
        const int mu = min(2, G.M - 2 * h);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (u < mu) {
                obstacle_terms<R, false, CLEAR>(G, sm, 2 * h + u, t, x[u], y[u], z[u], rr[u]);
                b[u] = x[u] * x[u] + y[u] * y[u] + z[u] * z[u] - rr[u] * rr[u];
            } else {
                x[u] = y[u] = z[u] = rr[u] = R(0);
                b[u] = R(1e30);
            }
        }
        for (int s = 0; s < G.S; ++s) {
            const R cx = px + sm[4 * s], cy = py + sm[4 * s + 1], cz = pz + sm[4 * s + 2], rs = sm[4 * s + 3];
            if constexpr (CLEAR) {
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    if (u < mu) {
                        const R dx = cx - x[u], dy = cy - y[u], dz = cz - z[u];
                        const R d2 = norm2(dx, dy, dz);
                        const R sum = rs + rr[u];
                        const R cl = rsqrt_r(d2) - sum;
                        val = cl < val ? cl : val;
                        hit = hit || (d2 < sum * sum);
                    }
                }
            } else if constexpr (sizeof(R) == 4) {
                const float thr = rs * (G.uniform_ro ? rs + 2.f * G.ro_uni : rs) - (cx * cx + cy * cy + cz * cz);
                unsigned long long v = ffma2(pk2(cx, cx), pk2(-2.f * x[0], -2.f * x[1]), pk2(b[0], b[1]));
                v = ffma2(pk2(cy, cy), pk2(-2.f * y[0], -2.f * y[1]), v);
                v = ffma2(pk2(cz, cz), pk2(-2.f * z[0], -2.f * z[1]), v);
                if (!G.uniform_ro) v = ffma2(pk2(rs, rs), pk2(-2.f * rr[0], -2.f * rr[1]), v);
                float lo, hi;
                upk2(v, lo, hi);
                const float e = fminf(lo, hi) - thr;
                val = fminf(val, e);
                hit = hit || e < 0.f;
            } else {
                const R negA = rs * rs - (cx * cx + cy * cy + cz * cz);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    R a = b[u];
                    a = cx * (R(-2) * x[u]) + a;
                    a = cy * (R(-2) * y[u]) + a;
                    a = cz * (R(-2) * z[u]) + a;
                    a = rs * (R(-2) * rr[u]) + a;
                    const R e = a - negA;
                    val = rmin(val, e);
                    hit = hit || e < R(0);
                }
            }
        }
    }
}

// edge_pool's smallest distance of an edge, order-encoded for atomicMin.
__device__ __forceinline__ void pool_best_reset(float& b) { *reinterpret_cast<int*>(&b) = ord_enc(rinf<float>()); }
__device__ __forceinline__ void pool_best_reset(double& b) {
    *reinterpret_cast<long long*>(&b) = ord_enc(rinf<double>());
}
__device__ __forceinline__ float pool_best_get(const float& b) {
    return ord_dec(*reinterpret_cast<const volatile int*>(&b));
}
__device__ __forceinline__ double pool_best_get(const double& b) {
    return ord_dec(*reinterpret_cast<const volatile long long*>(&b));
}

// What a warp works with: the blob and tables of the block, its own shared
// memory and its lane's joints.
template <typename R, int L>
struct WarpEdges {
    const float* smf;  // FP32 blob (arms)
    const R* blob;     // the problem's blob: a point robot's in shared memory, an FP64 arm's through the cache
    const int* sfr;    // frame of each sphere
    const float* reach;
    const R* tab;
    PointScratch P;
    float* lb;         // distance bound of each sphere
    R* xfr;            // frames and centres of the exact pass
    R* xsc;
    R th0[8 / L], qlo[8 / L], qhi[8 / L];
    int lane, r, grp;
    bool lip;
};

// Block-wide staging: the blob by one TMA bulk copy (unless staged) and the
// tables. Returns false when the copy's wait ran out.
template <typename R, bool ARM>
__device__ __forceinline__ bool edge_stage(const Geom<R>& G, const Geom<float>& GF, int* err, unsigned char* smem_raw,
                                           uint64_t* bar, bool staged) {
    // In shared memory: the FP32 blob of an arm, or a point robot's own.
    const unsigned blob_bytes = ARM ? GF.blob_bytes : G.blob_bytes;
    R* tab = reinterpret_cast<R*>(smem_raw + blob_bytes);  // [8][4]: th0, q_lo, q_hi
    float* reach = reinterpret_cast<float*>(smem_raw + blob_bytes + 4 * 8 * sizeof(R));  // [joint][frame]
    int* sfr = reinterpret_cast<int*>(reach + 64);
    if (!staged && threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, blob_bytes);
        bulk_g2s(smem_raw, ARM ? (const void*)GF.blob : (const void*)G.blob, blob_bytes, bar);
    }
    for (int i = threadIdx.x; i < 64; i += blockDim.x) {
        reach[i] = i < 8 * kMaxDof ? G.lip_reach[i] : 0.f;
        if (i < 8) {
            tab[4 * i] = i < G.dof ? G.th0[i] : R(0);
            tab[4 * i + 1] = i < G.dof ? G.qlo[i] : R(0);
            tab[4 * i + 2] = i < G.dof ? G.qhi[i] : R(0);
        }
    }
    if (ARM) {
        for (int s = threadIdx.x; s < G.S; s += blockDim.x) {
            int f = 0;
#pragma unroll
            for (int j = 1; j <= kMaxDof; ++j)
                if (j <= G.dof && s >= G.link_start[j]) f = j;
            sfr[s] = f;
        }
    }
    __syncthreads();
    if (!staged && !mbar_wait(bar, 0)) {
        if (threadIdx.x == 0 && err) atomicOr(err, kErrTimeout);
        return false;
    }
    return true;
}

template <typename R, bool ARM, bool EXACT, int L>
__device__ __forceinline__ void warp_edges(const Geom<R>& G, const Geom<float>& GF, unsigned char* smem_raw,
                                           unsigned char* wbase, const EdgeShared& lay, WarpEdges<R, L>& W) {
    constexpr int NP = 32 / L;
    const unsigned blob_bytes = ARM ? GF.blob_bytes : G.blob_bytes;
    W.smf = reinterpret_cast<const float*>(smem_raw);
    W.blob = ARM && sizeof(R) == 8 ? G.blob : reinterpret_cast<const R*>(smem_raw);
    W.tab = reinterpret_cast<const R*>(smem_raw + blob_bytes);
    W.reach = reinterpret_cast<const float*>(smem_raw + blob_bytes + 4 * 8 * sizeof(R));
    W.sfr = reinterpret_cast<const int*>(W.reach + 64);
    W.lane = threadIdx.x & 31;
    W.r = W.lane & (L - 1);
    W.grp = W.lane / L;
    W.lip = G.lip_ok && G.n_self == 0;
    W.lb = reinterpret_cast<float*>(wbase + lay.dist) + W.grp * kMaxSpheres;
    W.P.chunk = edge_chunk_of(G.M, L);
    float* t = reinterpret_cast<float*>(wbase + lay.near);
    const int os = edge_obs_stride(W.P.chunk);
    W.P.fr = t + W.grp * kFrameStride;
    W.P.ob = t + NP * kFrameStride + W.grp * os;
    W.P.ro = W.P.ob + 4 * W.P.chunk;
    W.P.sc = ARM && !EXACT && G.n_self > 0 ? t + NP * (kFrameStride + os) + W.grp * edge_self_stride(G.S) : nullptr;
    W.xfr = nullptr;
    W.xsc = nullptr;
    if constexpr (EXACT) {
        R* x = reinterpret_cast<R*>(wbase + lay.exact);
        if constexpr (sizeof(R) == 8) {
            W.xfr = x + W.grp * kFrameStride;
            x += NP * kFrameStride;
        } else {
            W.xfr = W.P.fr;  // the near pass's frames are the FP32 ones
        }
        if (G.n_self > 0) W.xsc = x + W.grp * edge_self_stride(G.S);
    }
#pragma unroll
    for (int i = 0; i < 8 / L; ++i) {
        W.th0[i] = W.tab[4 * (W.r + L * i)];
        W.qlo[i] = W.tab[4 * (W.r + L * i) + 1];
        W.qhi[i] = W.tab[4 * (W.r + L * i) + 2];
    }
}

// Check point s of each group's edge (joint j at lane j % L; have: the group has
// one). hit: the lane saw a collision; best: clearances, the group's smallest
// distance so far, updated; returns the check points to either side that this
// one decides. The warp runs it together.
template <typename R, bool ARM, bool CLEAR, int L>
__device__ __forceinline__ int edge_point(const Geom<R>& G, const Geom<float>& GF, const WarpEdges<R, L>& W, bool have,
                                          R s, const R (&qa)[8 / L], const R (&qb)[8 / L], R ta, R tb, float mu,
                                          bool cover, const float* dv, bool& hit, R& best) {
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool kExact = ARM && (CLEAR || sizeof(R) == 8);
    R q[8 / L];
#pragma unroll
    for (int i = 0; i < 8 / L; ++i) {
        q[i] = qa[i] + s * (qb[i] - qa[i]);
        hit = hit || (W.r + L * i < G.dof && ((q[i] < W.qlo[i]) || (q[i] > W.qhi[i])));
    }
    const R t = ta + s * (tb - ta);
    float steps = rinf<float>();
    if constexpr (ARM) {
        float th[8 / L], e32 = rinf<float>();
#pragma unroll
        for (int i = 0; i < 8 / L; ++i) th[i] = (float)(q[i] + W.th0[i]);
        near_pass<kExact, L>(GF, W.smf, W.sfr, W.P, dv, W.r, th, (float)t, mu, e32, steps, W.lb);
        if constexpr (!kExact) {
            hit = hit || e32 < 0.f;
            if (W.P.sc) {
                __syncwarp();
                float none = 0.f;
                self_pairs<float, false, L>(GF, W.smf, W.smf + GF.off_self, W.P.sc, W.r, hit, none);
            }
        }
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) steps = fminf(steps, __shfl_xor_sync(kFull, steps, o));
        __syncwarp();  // the scratch is rewritten below or by the next point
        if constexpr (kExact) {
            // steps: the smallest distance bound less the margin.
            R val = CLEAR ? best : R(0);
            const bool all = !G.lip_ok || !(mu < 1e30f);  // the bounds do not apply
            bool open = have && (!(steps > (float)val) || all || G.n_self > 0);
            if constexpr (!CLEAR) {
                // Deeper than the rounding of e and of the positions: a collision.
#pragma unroll
                for (int o = L / 2; o > 0; o >>= 1) e32 = fminf(e32, __shfl_xor_sync(kFull, e32, o));
                if (e32 < -2.f * G.lip_rr * mu - G.lip_eps && !all) {
                    hit = true;
                    open = false;
                }
            }
            if (__any_sync(kFull, open)) {
                const R* ob = nullptr;
                const R* ro = nullptr;
                if constexpr (sizeof(R) == 4) {
                    if (G.M <= W.P.chunk) {
                        ob = W.P.ob;
                        ro = W.P.ro;
                    }
                }
                exact_pass<R, CLEAR, L>(G, W.blob, W.sfr, W.xfr, ob, ro, W.xsc, W.lb, W.r, q[0] + W.th0[0], t, open, all,
                                        hit, val);
#pragma unroll
                for (int o = L / 2; o > 0; o >>= 1) val = rmin(val, __shfl_xor_sync(kFull, val, o));
                __syncwarp();
            }
            if constexpr (CLEAR) best = rmin(best, val);
            const float floor_d = CLEAR ? (float)best : 0.f;
            steps = rinf<float>();
            for (int k = W.r; k < G.S; k += L) steps = fminf(steps, (W.lb[k] - floor_d) * dv[W.sfr[k]]);
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) steps = fminf(steps, __shfl_xor_sync(kFull, steps, o));
            __syncwarp();
        }
    } else {
        R val = rinf<R>();
        point_robot<R, CLEAR, L>(G, W.blob, W.r, q[0], t, hit, val);
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) val = rmin(val, __shfl_xor_sync(kFull, val, o));
        if constexpr (CLEAR) {
            if (have) best = rmin(best, val);
            steps = ((float)(val - best) - mu) * dv[0];
        } else {
            steps = (sqrt_approx(fmaf(G.lip_rr, G.lip_rr, (float)val)) - G.lip_rr - mu) * dv[0];
        }
    }
    return cover ? (int)floor_steps(steps) : 0;
}

// smem_raw (both bodies): the blob, the tables, in edge_pool the pool, and the
// shared memory of nwarps warps (warps of the block beyond nwarps have no part
// in the batch). cta / ncta: this CTA among those sharing the batch. GF: the
// geometry in FP32 (G itself in FP32). Edges of count 0 are left out. E.next is
// zero at the launch.
//
// edge_stream: warps take their first block of `grab` consecutive edges by their
// number and later ones from E.next.
template <typename R, bool ARM, bool CLEAR, int L>
__device__ __forceinline__ void edge_stream(const Geom<R>& G, const Geom<float>& GF, const EdgeBatch<R>& E,
                                            unsigned char* smem_raw, int nwarps, int cta, int ncta, int grab) {
    constexpr int JL = 8 / L;  // joints per lane
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool kExact = ARM && (CLEAR || sizeof(R) == 8);
    static_assert(!kExact || L == 8, "the exact pass has a joint per lane");
    __shared__ __align__(8) uint64_t bar;
    const int n = E.n_host;
    if (!edge_stage<R, ARM>(G, GF, E.err, smem_raw, &bar, false)) return;
    const int warp = threadIdx.x >> 5;
    const EdgeShared lay = edge_shared<R>(ARM, G.S, G.M, G.n_self, L, false, kExact);
    unsigned char* wbase = smem_raw + (ARM ? GF.blob_bytes : G.blob_bytes) + edge_table_bytes<R>() +
                           (size_t)warp * lay.bytes;
    WarpEdges<R, L> W;
    warp_edges<R, ARM, kExact, L>(G, GF, smem_raw, wbase, lay, W);
    const int lane = W.lane, r = W.r, grp = W.grp;
    const unsigned grp_lanes = ((1u << L) - 1u) << (grp * L);
    int2* stack = reinterpret_cast<int2*>(wbase) + grp * kEdgeStack;
    float* dv = reinterpret_cast<float*>(wbase + lay.steps) + grp * 8;  // steps per metre by frame
    float* held = reinterpret_cast<float*>(wbase + lay.held);           // [32][kHeld]

    // Block of edges this warp holds: base, counts (lane i: edge base + i) and
    // the lanes whose edge is still to be taken.
    const int gw = cta * nwarps + warp, nw = ncta * nwarps;
    int base = 0, cnt_l = 0;
    unsigned pend = 0;
    bool first = true, more = true;
    // The group's edge.
    int e = -1, c = 0, depth = 0;
    R qa[JL], qb[JL], ta = R(0), tb = R(0);
#pragma unroll
    for (int i = 0; i < JL; ++i) qa[i] = qb[i] = R(0);
    float mu = 0.f;
    bool ehit = false;
    R best = rinf<R>();
    unsigned long long points = 0;

    for (;;) {
        // Groups without an edge take the next pending one.
        unsigned need = __ballot_sync(kFull, r == 0 && e < 0);
        while (need) {
            if (!pend && more) {
                long long b;
                if (first) {
                    b = (long long)gw * grab;
                    first = false;
                } else {
                    int v = 0;
                    if (lane == 0) v = atomicAdd(E.next, 1);
                    b = ((long long)nw + __shfl_sync(kFull, v, 0)) * grab;
                }
                if (b >= n) {
                    more = false;
                } else {
                    if ((long long)nw * grab >= n) more = false;  // every edge belongs to a first block
                    base = (int)b;
                    const int k = min(grab, n - base);
                    cnt_l = 0;
                    if (lane < k) {
                        // Lane i: edge base + i. Its count, the bound on the approach per check
                        // point by frame, and the margin.
                        const int i = base + lane;
                        R ra[kMaxDof], rb[kMaxDof];
                        const R t0 = E.ta[i], t1 = E.tb[i];
#pragma unroll
                        for (int j = 0; j < kMaxDof; ++j) {
                            ra[j] = j < G.dof ? E.qa[(size_t)i * E.qstride + j] : R(0);
                            rb[j] = j < G.dof ? E.qb[(size_t)i * E.qstride + j] : R(0);
                        }
                        cnt_l = E.cnt ? E.cnt[i] : edge_count<R>(ra, rb, t0, t1, G.dof, G.vmax_d, E.res);
                        bool in = true;
                        float dl[8], mg[8];
#pragma unroll
                        for (int f = 0; f < 8; ++f) dl[f] = mg[f] = 0.f;
#pragma unroll
                        for (int j = 0; j < kMaxDof; ++j) {
                            if (j < G.dof) {
                                const float qm = fabsf((float)ra[j]) + fabsf((float)rb[j]);
                                const float dq = fabsf((float)(rb[j] - ra[j]));
                                const float bt = box_margin(qm);
                                const R lo = W.tab[4 * j + 1], hi = W.tab[4 * j + 2];
                                in = in && (float)(ra[j] - lo) > bt && (float)(hi - ra[j]) > bt &&
                                     (float)(rb[j] - lo) > bt && (float)(hi - rb[j]) > bt;
#pragma unroll
                                for (int f = 0; f < 8; ++f) {
                                    dl[f] = fmaf(dq, W.reach[8 * j + f], dl[f]);
                                    mg[f] = fmaf(qm, W.reach[8 * j + f], mg[f]);
                                }
                            }
                        }
                        const float dt = G.lip_v * fabsf((float)(t1 - t0));
                        float m = 0.f;
#pragma unroll
                        for (int f = 0; f < 8; ++f) {
                            m = fmaxf(m, mg[f]);
                            held[kHeld * lane + f] = (float)cnt_l / ((dl[f] + dt) * 1.00002f);
                        }
                        m += G.lip_v * (fabsf((float)t0) + fabsf((float)t1));
                        held[kHeld * lane + 8] = G.lip_mu + 1e-6f * m;
                        int2 box = make_int2(0, cnt_l);
                        if (!in) {
                            float s1 = 0.f, s2 = 1.f;
#pragma unroll
                            for (int j = 0; j < kMaxDof; ++j)
                                if (j < G.dof) box_joint<R>(ra[j], rb[j], W.tab[4 * j + 1], W.tab[4 * j + 2], s1, s2);
                            box = box_range(s1, s2, cnt_l);
                        }
                        if (!(W.lip && m < 1e6f)) box = make_int2(0, 0);
                        held[kHeld * lane + 9] = __int_as_float(box.x);
                        held[kHeld * lane + 10] = __int_as_float(box.y);
                        if (E.n_checks) E.n_checks[i] = cnt_l;
                        if (!E.cnt && cnt_l <= 0) {  // no check point (a length that is not a number)
                            if (E.verdict) E.verdict[i] = 1;
                            if (CLEAR && E.clear) E.clear[i] = rinf<R>();
                        }
                    }
                    pend = __ballot_sync(kFull, cnt_l > 0);
                    __syncwarp();  // other lanes read this lane's bounds
                }
                if (!pend) {
                    if (!more) break;
                    continue;
                }
            }
            if (!pend) break;
            // The k-th needing group takes the k-th pending edge.
            int src = -1;
            {
                unsigned p = pend, q = need;
                while (p && q) {
                    const int tl = __ffs(q) - 1, pl = __ffs(p) - 1;
                    if ((grp_lanes >> tl) & 1u) src = pl;
                    p &= p - 1;
                    q &= q - 1;
                }
                pend = p;
                need = q;
            }
            const int cc = __shfl_sync(kFull, cnt_l, src < 0 ? 0 : src);
            if (src >= 0) {
                e = base + src;
                c = cc;
                const size_t row = (size_t)e * E.qstride;
#pragma unroll
                for (int i = 0; i < JL; ++i) {
                    const int j = r + L * i;
                    qa[i] = j < G.dof ? E.qa[row + j] : R(0);
                    qb[i] = j < G.dof ? E.qb[row + j] : R(0);
                }
                ta = E.ta[e];
                tb = E.tb[e];
                ehit = false;
                best = rinf<R>();
                for (int f = r; f < 8; f += L) dv[f] = held[kHeld * src + f];
                mu = held[kHeld * src + 8];
                const int x = __float_as_int(held[kHeld * src + 9]), y = __float_as_int(held[kHeld * src + 10]);
                depth = 0;
                auto push = [&](int lo, int last, bool covers) {
                    if (lo > last) return;
                    if (r == 0) stack[depth] = make_int2(lo, covers ? last : -last);
                    ++depth;
                };
                push(x + 1, y, true);
                push(1, x, false);
                push(y + 1, c, false);
            }
            __syncwarp();
        }
        if (!__any_sync(kFull, e >= 0)) break;

        // Each group takes an interval and evaluates its middle (its first
        // point when the stack is nearly full, which leaves one interval).
        const bool have = e >= 0;
        int lo = 1, hi = 0, m = 1;
        bool covers = false;
        if (have) {
            const int2 iv = stack[depth - 1];
            lo = iv.x;
            hi = abs(iv.y);
            covers = iv.y > 0;
            m = depth + 1 > kEdgeStack ? lo : lo + ((hi - lo) >> 1);
            --depth;
            if (r == 0) ++points;
        }
        __syncwarp();  // the interval's slot may be rewritten below
        bool hit = false;
        const int far = edge_point<R, ARM, CLEAR, L>(G, GF, W, have, R(m) / R(c > 0 ? c : 1), qa, qb, ta, tb, mu,
                                                     covers, dv, hit, best);
        const unsigned hits = __ballot_sync(kFull, have && hit);  // every lane takes part
        ehit = ehit || (hits & grp_lanes) != 0;
        // What the point does not decide goes back, unless the edge is decided.
        if (have && (CLEAR || !ehit)) {
            if (far < m - lo) {
                if (r == 0) stack[depth] = make_int2(lo, covers ? m - 1 - far : 1 - m);
                ++depth;
            }
            if (far < hi - m) {
                if (r == 0) stack[depth] = make_int2(m + 1 + far, covers ? hi : -hi);
                ++depth;
            }
        }
        if (have && ((!CLEAR && ehit) || depth == 0)) {
            if (r == 0) {
                if (E.verdict) E.verdict[e] = ehit ? 0 : 1;
                if (E.hit && ehit) E.hit[e] = 1;
                if (CLEAR && E.clear) E.clear[e] = best;
            }
            e = -1;
            depth = 0;
        }
        __syncwarp();
    }
    if (E.points_done || E.pairs_done) {
        for (int o = 16; o > 0; o >>= 1) points += __shfl_xor_sync(kFull, points, o);
        if (lane == 0 && points) {
            if (E.points_done) atomicAdd(E.points_done, points);
            if (E.pairs_done) atomicAdd(E.pairs_done, points * (unsigned long long)(G.S * G.M));
        }
    }
}

// edge_pool: a CTA takes `edges` consecutive edges (the first block by its
// number, later ones from E.next), splits each into `pieces` intervals and
// evaluates the middles of all undecided intervals, level by level.
template <typename R, bool ARM, bool CLEAR>
__device__ __forceinline__ void edge_pool(const Geom<R>& G, const Geom<float>& GF, const EdgeBatch<R>& E,
                                          unsigned char* smem_raw, int nwarps, int cta, int ncta, int edges, int pieces,
                                          bool staged) {
    constexpr int L = kPoolLanes, NP = 32 / L;
    constexpr unsigned kFull = 0xffffffffu;
    constexpr bool kExact = ARM && (CLEAR || sizeof(R) == 8);
    static_assert(L == 8, "a joint and a frame per lane");
    __shared__ __align__(8) uint64_t bar;
    const int n = E.n_host;
    if (n <= 0 || (E.done && *E.done)) return;
    if (!edge_stage<R, ARM>(G, GF, E.err, smem_raw, &bar, staged)) return;
    const unsigned head = (ARM ? GF.blob_bytes : G.blob_bytes) + edge_table_bytes<R>();
    PoolShared<R>& S = *reinterpret_cast<PoolShared<R>*>(smem_raw + head);
    const int warp = threadIdx.x >> 5;
    const bool works = warp < nwarps;
    const EdgeShared lay = edge_shared<R>(ARM, G.S, G.M, G.n_self, L, true, kExact);
    WarpEdges<R, L> W;
    warp_edges<R, ARM, kExact, L>(G, GF, smem_raw, smem_raw + head + pool_bytes<R>() + (size_t)(works ? warp : 0) * lay.bytes,
                                  lay, W);
    const int lane = W.lane, r = W.r, grp = W.grp;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned grp_lanes = ((1u << L) - 1u) << (grp * L);
    unsigned points = 0;

    for (int wave = 0;; ++wave) {
        if (threadIdx.x == 0) {
            S.base = wave == 0 ? (long long)cta * edges : ((long long)ncta + atomicAdd(E.next, 1)) * edges;
            S.n[0] = S.n[1] = S.n[2] = 0;
            S.nslot = 0;
        }
        __syncthreads();
        const long long base = S.base;
        if (base >= n) break;
        const int k = (int)min((long long)edges, n - base);
        // A group per edge: endpoints, count, bounds and the first intervals.
        for (int i0 = warp * NP; works && i0 < k; i0 += nwarps * NP) {
            const int i = i0 + grp;
            const int e = (int)base + (i < k ? i : 0);
            const size_t row = (size_t)e * E.qstride;
            const R qa = r < G.dof ? E.qa[row + r] : R(0), qb = r < G.dof ? E.qb[row + r] : R(0);
            const R ta = E.ta[e], tb = E.tb[e];
            const float qm = fabsf((float)qa) + fabsf((float)qb), dq = fabsf((float)(qb - qa));
            int c;
            if (E.cnt) {
                c = E.cnt[e];
            } else {
                // Every lane forms the row (the count is that of edge_count).
                R ra[kMaxDof], rb[kMaxDof];
#pragma unroll
                for (int j = 0; j < kMaxDof; ++j) {
                    ra[j] = __shfl_sync(kFull, qa, j, L);
                    rb[j] = __shfl_sync(kFull, qb, j, L);
                }
                c = edge_count<R>(ra, rb, ta, tb, G.dof, G.vmax_d, E.res);
            }
            const float bt = box_margin(qm);
            const bool in = r >= G.dof || c <= 0 ||
                            ((float)(qa - W.qlo[0]) > bt && (float)(W.qhi[0] - qa) > bt &&
                             (float)(qb - W.qlo[0]) > bt && (float)(W.qhi[0] - qb) > bt);
            float dl = 0.f, mg = 0.f;  // lane r: frame r
#pragma unroll
            for (int j = 0; j < kMaxDof; ++j) {
                const float a = W.reach[8 * j + r];
                dl = fmaf(__shfl_sync(kFull, dq, j, L), a, dl);
                mg = fmaf(__shfl_sync(kFull, qm, j, L), a, mg);
            }
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) mg = fmaxf(mg, __shfl_xor_sync(kFull, mg, o));
            mg += G.lip_v * (fabsf((float)ta) + fabsf((float)tb));
            int2 box = make_int2(0, c);
            if (__any_sync(kFull, !in)) {
                float s1 = 0.f, s2 = 1.f;
                if (!in) box_joint<R>(qa, qb, W.qlo[0], W.qhi[0], s1, s2);
#pragma unroll
                for (int o = L / 2; o > 0; o >>= 1) {
                    s1 = fmaxf(s1, __shfl_xor_sync(kFull, s1, o));
                    s2 = fminf(s2, __shfl_xor_sync(kFull, s2, o));
                }
                if (s1 > 0.f || s2 < 1.f) box = box_range(s1, s2, c);
            }
            int slot = -1, at = 0;
            // The stretch that is cut into pieces: the covered one, or the whole edge.
            const int px = box.x, py = box.y > 0 ? box.y : c;
            const int np = min(pieces, py - px);
            if (r == 0 && i < k) {
                if (E.n_checks) E.n_checks[e] = c;
                if (c > 0) {
                    slot = atomicAdd(&S.nslot, 1);
                    at = atomicAdd(&S.n[0], np + (px > 0) + (py < c));
                } else if (!E.cnt) {  // no check point (a length that is not a number)
                    if (E.verdict) E.verdict[e] = 1;
                    if (CLEAR && E.clear) E.clear[e] = rinf<R>();
                }
            }
            slot = __shfl_sync(kFull, slot, 0, L);
            at = __shfl_sync(kFull, at, 0, L);
            if (slot >= 0) {
                S.q[slot][r] = qa;
                S.q[slot][8 + r] = qb;
                S.dv[slot][r] = (float)c / ((dl + G.lip_v * fabsf((float)(tb - ta))) * 1.00002f);
                if (r == 0) {
                    S.t[slot][0] = ta;
                    S.t[slot][1] = tb;
                    S.mu[slot] = G.lip_mu + 1e-6f * mg;
                    S.c[slot] = c;
                    S.edge[slot] = e;
                    S.hit[slot] = 0;
                    pool_best_reset(S.best[slot]);
                }
                for (int g = r; g < np; g += L) {
                    const bool covers = box.y > 0 && W.lip && mg < 1e6f;
                    const int last = px + (int)((long long)(py - px) * (g + 1) / np);
                    S.iv[0][at + g] = make_int2(px + 1 + (int)((long long)(py - px) * g / np), covers ? last : -last);
                    S.slot[0][at + g] = (unsigned char)slot;
                }
                if (r == 0 && px > 0) {
                    S.iv[0][at + np] = make_int2(1, -px);
                    S.slot[0][at + np] = (unsigned char)slot;
                }
                if (r == 0 && py < c) {
                    S.iv[0][at + np + (px > 0)] = make_int2(py + 1, -c);
                    S.slot[0][at + np + (px > 0)] = (unsigned char)slot;
                }
            }
        }
        __syncthreads();
        // Levels: list `cur` is evaluated, the next one filled; the third
        // counter is cleared meanwhile.
        for (int level = 1;; ++level) {
            const int cur = (level - 1) % 3, nxt = level % 3, buf = (level - 1) & 1;
            const int nc = S.n[cur];
            if (nc == 0) break;
            if (threadIdx.x == 0) S.n[(level + 1) % 3] = 0;
            const bool single = 2 * nc > kPoolList;  // an interval leaves at most one
            for (int i0 = warp * NP; works && i0 < nc; i0 += nwarps * NP) {
                const int i = i0 + grp;
                int slot = 0, lo = 1, hi = 0, m = 1;
                bool have = i < nc, covers = false;
                if (have) {
                    const int2 iv = S.iv[buf][i];
                    slot = S.slot[buf][i];
                    lo = iv.x;
                    hi = abs(iv.y);
                    covers = iv.y > 0;
                    m = single ? lo : lo + ((hi - lo) >> 1);
                    const int h = *(volatile int*)&S.hit[slot];
                    have = CLEAR || h == 0 || h >= level;  // decided in an earlier level: nothing left to do
                }
                if (!__any_sync(kFull, have)) continue;
                const R qa[1] = {S.q[slot][r]}, qb[1] = {S.q[slot][8 + r]};
                R best = rinf<R>();
                if constexpr (CLEAR) best = pool_best_get(S.best[slot]);
                bool hit = false;
                const int far = edge_point<R, ARM, CLEAR, L>(G, GF, W, have, R(m) / R(S.c[slot]), qa, qb, S.t[slot][0],
                                                             S.t[slot][1], S.mu[slot], covers, S.dv[slot], hit,
                                                             best);
                const bool ghit = (__ballot_sync(kFull, have && hit) & grp_lanes) != 0;
                if (have && r == 0) {
                    ++points;
                    if (ghit && *(volatile int*)&S.hit[slot] == 0) *(volatile int*)&S.hit[slot] = level;
                    if constexpr (CLEAR) atomic_min_r<R>(&S.best[slot], best);
                }
                // What the point does not decide goes to the next level.
                const bool live = have && (CLEAR || !ghit);
                const bool left = live && far < m - lo, right = live && far < hi - m;
                const unsigned bl = __ballot_sync(kFull, left && r == 0), br = __ballot_sync(kFull, right && r == 0);
                int at = 0;
                if (lane == 0 && (bl | br)) at = atomicAdd(&S.n[nxt], __popc(bl) + __popc(br));
                at = __shfl_sync(kFull, at, 0) + __popc(bl & lt) + __popc(br & lt);
                if (r == 0) {
                    if (left) {
                        S.iv[buf ^ 1][at] = make_int2(lo, covers ? m - 1 - far : 1 - m);
                        S.slot[buf ^ 1][at] = (unsigned char)slot;
                        ++at;
                    }
                    if (right) {
                        S.iv[buf ^ 1][at] = make_int2(m + 1 + far, covers ? hi : -hi);
                        S.slot[buf ^ 1][at] = (unsigned char)slot;
                    }
                }
            }
            __syncthreads();
        }
        for (int i = threadIdx.x; i < S.nslot; i += blockDim.x) {
            const int e = S.edge[i];
            const bool h = S.hit[i] != 0;
            if (E.verdict) E.verdict[e] = h ? 0 : 1;
            if (E.hit && h) E.hit[e] = 1;
            if (CLEAR && E.clear) E.clear[e] = pool_best_get(S.best[i]);
        }
        if ((long long)ncta * edges >= n) break;  // every edge belongs to a first block
        __syncthreads();
    }
    if (E.points_done || E.pairs_done) {
        for (int o = 16; o > 0; o >>= 1) points += __shfl_xor_sync(kFull, points, o);
        if (lane == 0 && points) {
            if (E.points_done) atomicAdd(E.points_done, (unsigned long long)points);
            if (E.pairs_done) atomicAdd(E.pairs_done, (unsigned long long)points * (unsigned long long)(G.S * G.M));
        }
    }
}

}  // namespace stp
