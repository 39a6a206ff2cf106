// Collision-kernel launches: the stand-alone edge batch (stp_check_edges),
// the planner's per-step launches and the batched form, plus the flat-batch
// helpers (check counts, prefix sums, fills). The device code lives in
// stp_edges_body.cuh (bounded motion) and stp_validate_body.cuh (every point).
#include <algorithm>

#include "stp_edges_body.cuh"

namespace stp {

int validate_grid_blocks() {
    static std::mutex mu;
    static int sms[kMaxDevices] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 1;
    std::lock_guard<std::mutex> lock(mu);
    if (sms[dev] == 0) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms[dev] = n > 0 ? n : 1;
    }
    return sms[dev];
}

// Resident CTAs per SM of a kernel at a block size and shared-memory size: the
// last answer per device is kept (a process asks for few sizes).
struct Occupancy {
    std::mutex mu;
    int threads[kMaxDevices] = {}, smem[kMaxDevices] = {}, ctas[kMaxDevices] = {};
};
static cudaError_t resident_ctas(const void* kern, Occupancy& o, int threads, int smem, int* ctas) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(o.mu);
    if (o.ctas[dev] == 0 || o.threads[dev] != threads || o.smem[dev] != smem) {
        int b = 0;
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kern, threads, smem);
        if (e != cudaSuccess) return e;
        o.threads[dev] = threads;
        o.smem[dev] = smem;
        o.ctas[dev] = b < 1 ? 1 : b;
    }
    *ctas = o.ctas[dev];
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Bounded-motion validation.
// ---------------------------------------------------------------------------
constexpr int kEdgeWarps = 8;  // most warps of a CTA

// Lanes per check point of a kernel.
template <typename R, bool ARM, bool CLEAR, bool POOL>
constexpr int kEdgeLanes = POOL || (ARM && (CLEAR || sizeof(R) == 8)) ? kPoolLanes : kStreamLanes;

// take: edges a CTA (POOL) or a warp takes at a time. CTAS: resident on an SM by
// registers; two for clearances where shared memory holds no more (an arm among
// many obstacles), which spares the spills of 80 registers (clearances of 10,000
// arm7 edges among 64 obstacles 943 -> 887 us; where three fit, 20,000 UR5e edges
// among 16, two take 391 instead of 347).
template <bool ARM, bool CLEAR, bool POOL, int CTAS>
__global__ void __launch_bounds__(32 * kEdgeWarps, CTAS)
    k_edges(const __grid_constant__ Geom<float> G, const __grid_constant__ EdgeBatch<float> E, int take) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (POOL)
        edge_pool<float, ARM, CLEAR>(G, G, E, smem_raw, blockDim.x >> 5, blockIdx.x, gridDim.x, take, pool_pieces(take),
                                     false);
    else
        edge_stream<float, ARM, CLEAR, kEdgeLanes<float, ARM, CLEAR, POOL>>(G, G, E, smem_raw, blockDim.x >> 5,
                                                                            blockIdx.x, gridDim.x, take);
}
template <bool ARM, bool CLEAR, bool POOL>
__global__ void __launch_bounds__(32 * kEdgeWarps, 2)
    k_edges64(const __grid_constant__ Geom<double> G, const __grid_constant__ Geom<float> GF,
              const __grid_constant__ EdgeBatch<double> E, int take) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if constexpr (POOL)
        edge_pool<double, ARM, CLEAR>(G, GF, E, smem_raw, blockDim.x >> 5, blockIdx.x, gridDim.x, take, pool_pieces(take),
                                      false);
    else
        edge_stream<double, ARM, CLEAR, kEdgeLanes<double, ARM, CLEAR, POOL>>(G, GF, E, smem_raw, blockDim.x >> 5,
                                                                              blockIdx.x, gridDim.x, take);
}

// Batched planner form: problem blockIdx.y; its geometry and state are staged
// in shared memory, its extension (which = 0) or bridge (which = 1) edge
// entries are validated; arm vs point robot is chosen per problem.
template <typename R>
__global__ void __launch_bounds__(32 * kEdgeWarps, sizeof(R) == 4 ? 3 : 2)
    k_validate_batch(const Geom<R>* __restrict__ Gs, const State<R>* __restrict__ Ss, int which) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ Geom<R> G;
    __shared__ State<R> S;
    stage_problem(Gs, Ss, blockIdx.y, G, S);
    const EdgeBatch<R> E = which == 0 ? ext_batch(S) : bridge_batch(S);
    const int edges = pool_edges(E.n_host, gridDim.x);
    if (G.arm)
        edge_pool<R, true, false>(G, G, E, smem_raw, kEdgeWarps, blockIdx.x, gridDim.x, edges, pool_pieces(edges), false);
    else
        edge_pool<R, false, false>(G, G, E, smem_raw, kEdgeWarps, blockIdx.x, gridDim.x, edges, pool_pieces(edges), false);
}

static int edge_smem(unsigned blob_bytes, int block, const EdgeShared& l, int nwarps) {
    return (int)blob_bytes + block + nwarps * l.bytes;
}
template <typename R>
int edge_smem_bytes(const Geom<R>& g, const Geom<float>& gf, int nwarps) {
    return edge_smem(g.arm ? gf.blob_bytes : g.blob_bytes, edge_table_bytes<R>() + pool_bytes<R>(),
                     edge_shared<R>(g.arm, g.S, g.M, g.n_self, kPoolLanes, true, g.arm && sizeof(R) == 8), nwarps);
}
template int edge_smem_bytes<float>(const Geom<float>&, const Geom<float>&, int);
template int edge_smem_bytes<double>(const Geom<double>&, const Geom<float>&, int);

// Whether check points of a problem's edges can be left out at all.
template <typename R>
static bool bounded(const Geom<R>& g) { return g.lip_ok && g.n_self == 0; }

template <typename R, bool ARM, bool CLEAR, bool POOL, int CTAS>
static cudaError_t launch_edges_ctas(const Geom<R>& g, const Geom<float>& gf, const EdgeBatch<R>& e, int take,
                                     int warps, int smem, cudaStream_t st) {
    const void* kern;
    if constexpr (sizeof(R) == 4) kern = (const void*)k_edges<ARM, CLEAR, POOL, CTAS>;
    else kern = (const void*)k_edges64<ARM, CLEAR, POOL>;
    static SmemAttr attr;
    static Occupancy occ;
    cudaError_t err = ensure_smem(kern, attr, smem);
    if (err != cudaSuccess) return err;
    int ctas = 1;
    err = resident_ctas(kern, occ, 32 * warps, smem, &ctas);
    if (err != cudaSuccess) return err;
    const int resident = validate_grid_blocks() * ctas;
    if (POOL && take <= 0) {
        take = pool_edges(e.n_host, resident);
        // A free edge without a bound takes many times a colliding one's points: up to
        // eight edges a CTA are taken in halves, the second as CTAs come free (UR5e with
        // self-collision: 1,000 edges 78 -> 66 us, of up to 1,000 points 370 -> 220, a
        // plan of 1,024 workers 2.57 -> 2.25 ms; at eleven a CTA 144 -> 162 us).
        if (!bounded(g) && take <= 8) take = (take + 1) / 2;
    }
    const long long takes = ((long long)e.n_host + take - 1) / take;
    const int grid = (int)std::min<long long>(POOL ? takes : (takes + warps - 1) / warps, resident);
    if constexpr (sizeof(R) == 4) k_edges<ARM, CLEAR, POOL, CTAS><<<grid, 32 * warps, smem, st>>>(g, e, take);
    else k_edges64<ARM, CLEAR, POOL><<<grid, 32 * warps, smem, st>>>(g, gf, e, take);
    return cudaGetLastError();
}

// Eight warps to a CTA, fewer when their shared memory does not fit. take <= 0
// (POOL): the edges spread over the resident CTAs.
template <typename R, bool ARM, bool CLEAR, bool POOL>
static cudaError_t launch_edges(const Geom<R>& g, const Geom<float>& gf, const EdgeBatch<R>& e, int take,
                                cudaStream_t st) {
    constexpr int kMaxSmem = 224 * 1024, kSmSmem = 228 * 1024, kCtaSmem = 1024 + 64;  // reserved and static, a CTA
    const EdgeShared lay = edge_shared<R>(ARM, g.S, g.M, g.n_self, kEdgeLanes<R, ARM, CLEAR, POOL>, POOL,
                                          ARM && (CLEAR || sizeof(R) == 8));
    const unsigned blob = ARM ? gf.blob_bytes : g.blob_bytes;
    const int block = edge_table_bytes<R>() + (POOL ? pool_bytes<R>() : 0);
    int warps = kEdgeWarps;
    while (warps > 1 && edge_smem(blob, block, lay, warps) > kMaxSmem) --warps;
    const int smem = edge_smem(blob, block, lay, warps);
    if constexpr (sizeof(R) == 4 && ARM && CLEAR) {
        if (3 * (smem + kCtaSmem) <= kSmSmem)
            return launch_edges_ctas<R, ARM, CLEAR, POOL, 3>(g, gf, e, take, warps, smem, st);
        return launch_edges_ctas<R, ARM, CLEAR, POOL, 2>(g, gf, e, take, warps, smem, st);
    } else {
        return launch_edges_ctas<R, ARM, CLEAR, POOL, 3>(g, gf, e, take, warps, smem, st);
    }
}

template <typename R, bool CLEAR, bool POOL>
static cudaError_t launch_edges_of(const Geom<R>& g, const Geom<float>& gf, const EdgeBatch<R>& e, int take,
                                   cudaStream_t st) {
    return g.arm ? launch_edges<R, true, CLEAR, POOL>(g, gf, e, take, st)
                 : launch_edges<R, false, CLEAR, POOL>(g, gf, e, take, st);
}

// Pool or stream, by edges per SM. The stream has no barriers but ends with the
// few edges that need many points, each on one lane group: 150 us of the UR5e's,
// 550 us of the seven-axis arm's. The pool spreads those over a CTA, but its
// levels idle warps. Measured on 152 SMs, pool / stream, us: UR5e, 16 obstacles,
// 20,000 edges 71 / 183, 80,000 189 / 230, 160,000 345 / 282, 10^6 1990 / 727;
// arm7, 64 obstacles, 65,536 603 / 857, 131,072 1139 / 1044; clearances of 40,000
// 2971 / 4618, UR5e 80,000 1227 / 1524; FP64, 20,000 572 / 738, 60,000 1506 / 1091;
// two-joint point robot, 10,000 34 / 36, 40,000 57 / 44.
template <typename R>
static int pool_limit(int arm) { return !arm ? 96 : sizeof(R) == 4 ? 704 : 224; }
// Clearances without a bound need every point; in FP32, arms, above 264 edges an
// SM, the every-point kernel is the faster one (UR5e with self-collision, pool /
// every point, us: 20,000 edges 1291 / 1322, 60,000 3503 / 3355, 400,000 22800 /
// 21200; FP64, 60,000, 35.9 / 97.4 ms).
template <typename R>
bool clears_every_point(const Geom<R>& g, int n) {
    return sizeof(R) == 4 && g.arm && !bounded(g) && (long long)n > 264ll * validate_grid_blocks();
}
template bool clears_every_point<float>(const Geom<float>&, int);
template bool clears_every_point<double>(const Geom<double>&, int);
// planner: the batch's size is the planner's worker count; always the pool.
template <typename R>
cudaError_t launch_validate(const Geom<R>& g, const Geom<float>& gf, const EdgeBatch<R>& e, bool clearance,
                            bool planner, cudaStream_t st) {
    if (e.n_host <= 0) return cudaSuccess;
    if (planner) return launch_edges_of<R, false, true>(g, gf, e, 0, st);
    const int spread = (e.n_host + validate_grid_blocks() - 1) / validate_grid_blocks();  // edges per SM
    // Without the bound every point of an edge is evaluated (self-collision pairs,
    // geometry beyond the margins): the pool spreads them over the CTA at any size.
    // UR5e with self-collision, pool / stream: 200,000 edges 3.35 / 5.66 ms, 120,000
    // of up to 1,000 points 2.3 / 37.8 ms (their tail: an edge to a lane group).
    if (spread <= pool_limit<R>(g.arm) || !bounded(g))
        return clearance ? launch_edges_of<R, true, true>(g, gf, e, 0, st)
                         : launch_edges_of<R, false, true>(g, gf, e, 0, st);
    const int take = std::max(4, std::min(32, spread / (3 * kEdgeWarps * 4)));
    return clearance ? launch_edges_of<R, true, false>(g, gf, e, take, st)
                     : launch_edges_of<R, false, false>(g, gf, e, take, st);
}

// P <= 0 only sets the kernel's shared-memory attribute (nothing is launched).
template <typename R>
cudaError_t launch_validate_batch(const Geom<R>* Gs, const State<R>* Ss, int P, int which, int ctas_per_problem,
                                  int smem_bytes, cudaStream_t st) {
    auto kern = k_validate_batch<R>;
    static SmemAttr attr;
    cudaError_t err = ensure_smem((const void*)kern, attr, smem_bytes);
    if (err != cudaSuccess) return err;
    if (P <= 0) return cudaSuccess;
    kern<<<dim3(ctas_per_problem, P), 32 * kEdgeWarps, smem_bytes, st>>>(Gs, Ss, which);
    return cudaGetLastError();
}
template cudaError_t launch_validate_batch<float>(const Geom<float>*, const State<float>*, int, int, int, int,
                                                  cudaStream_t);

// ---------------------------------------------------------------------------
// Every-point validation.
// ---------------------------------------------------------------------------
template <typename R, bool ARM, int MO, bool CLEAR>
__global__ void __launch_bounds__(256, (sizeof(R) == 4 && MO <= 16) ? 2 : 1)
    k_validate_full(const __grid_constant__ Geom<R> G, const __grid_constant__ EdgeBatch<R> E) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    validate_full_body<R, ARM, MO, CLEAR>(G, E, smem_raw);
}

template <typename R, bool ARM, int MO, bool CLEAR>
static cudaError_t launch_full(const Geom<R>& g, const EdgeBatch<R>& e, cudaStream_t st) {
    auto kern = k_validate_full<R, ARM, MO, CLEAR>;
    static SmemAttr attr;
    static Occupancy occ;
    const int smem = (int)g.blob_bytes + (int)(sizeof(long long) * (kWin + 1));
    cudaError_t err = ensure_smem((const void*)kern, attr, smem);
    if (err != cudaSuccess) return err;
    int ctas = 1;
    err = resident_ctas((const void*)kern, occ, 256, smem, &ctas);
    if (err != cudaSuccess) return err;
    const int grid = validate_grid_blocks() * ctas;
    kern<<<grid, 256, smem, st>>>(g, e);
    return cudaGetLastError();
}

// Obstacle chunk per pass: FP32 keeps at most 16 obstacles in registers
// (128 registers, two CTAs per SM; more obstacles take more passes, each
// repeating the forward kinematics), FP64 up to 32.
template <typename R, bool ARM>
static cudaError_t launch_full_mo(const Geom<R>& g, const EdgeBatch<R>& e, cudaStream_t st) {
    if (g.M <= 8) return launch_full<R, ARM, 8, false>(g, e, st);
    if constexpr (sizeof(R) == 4) {
        return launch_full<R, ARM, 16, false>(g, e, st);
    } else {
        if (g.M <= 16) return launch_full<R, ARM, 16, false>(g, e, st);
        return launch_full<R, ARM, 32, false>(g, e, st);
    }
}
// clearance: 16 obstacles at a time in either precision (their coordinates and
// radii stay apart in the direct form, so 32 would not fit the registers).
template <typename R>
cudaError_t launch_validate_full(const Geom<R>& g, const EdgeBatch<R>& e, bool clearance, cudaStream_t st) {
    if (clearance) return g.arm ? launch_full<R, true, 16, true>(g, e, st) : launch_full<R, false, 16, true>(g, e, st);
    return g.arm ? launch_full_mo<R, true>(g, e, st) : launch_full_mo<R, false>(g, e, st);
}

// ---------------------------------------------------------------------------
// Closed-form (continuous) validation of point-robot edges, one lane per
// edge. Between consecutive breakpoints (the edge's end times and each
// obstacle waypoint time inside them) a robot sphere and an obstacle both
// move linearly, so their difference runs along the segment from d(t0) to
// d(t1) and its smallest norm is the distance from the origin to that segment.
// A pair collides iff that squared minimum < (r + r_o)^2; the edge stays in
// the convex configuration box iff both ends do.
// ---------------------------------------------------------------------------
template <typename R, bool CLEAR>
__global__ void __launch_bounds__(256) k_validate_cont(Geom<R> G, EdgeBatch<R> E) {
    const int n = E.n_host;
    if (n <= 0 || (E.done && *E.done)) return;
    const R* sph = G.blob;
    const R* way = G.blob + G.off_way;
    const R* vel = G.blob + G.off_vel;
    const R* rad = G.blob + G.off_rad;
    unsigned long long done = 0, pairs_total = 0;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
        if (E.cnt[e] <= 0) continue;
        const R* qa = E.qa + (size_t)e * E.qstride;
        const R* qb = E.qb + (size_t)e * E.qstride;
        const R ta = E.ta[e], tb = E.tb[e];
        bool hit = false;
        for (int j = 0; j < G.dof; ++j)
            hit = hit || qa[j] < G.qlo[j] || qa[j] > G.qhi[j] || qb[j] < G.qlo[j] || qb[j] > G.qhi[j];
        const R pa[3] = {qa[0], qa[1], G.dof > 2 ? qa[2] : R(0)};
        const R pb[3] = {qb[0], qb[1], G.dof > 2 ? qb[2] : R(0)};
        R clr = rinf<R>();
        for (int m = 0; m < G.M; ++m) {
            const R* W = way + 4 * G.K * m;
            const R* V = vel + 4 * G.K * m;
            const R ro = rad[m];
            R t0 = ta;
            for (int k = 0; k <= G.K; ++k) {
                // next breakpoint: waypoint k if inside (ta, tb), the end at k == K
                R t1;
                if (k < G.K) {
                    t1 = W[4 * k];
                    if (!(t1 > ta && t1 < tb)) continue;
                } else {
                    t1 = tb;
                }
                const R f0 = tb > ta ? (t0 - ta) / (tb - ta) : R(0);
                const R f1 = tb > ta ? (t1 - ta) / (tb - ta) : R(0);
                R o0[3], o1[3];
                obstacle_at(W, V, G.K, t0, o0[0], o0[1], o0[2]);
                obstacle_at(W, V, G.K, t1, o1[0], o1[1], o1[2]);
                for (int sp = 0; sp < G.S; ++sp) {
                    R d0[3], w[3];
                    for (int i = 0; i < 3; ++i) {
                        const R c0 = (pa[i] + f0 * (pb[i] - pa[i])) + sph[4 * sp + i];
                        const R c1 = (pa[i] + f1 * (pb[i] - pa[i])) + sph[4 * sp + i];
                        d0[i] = c0 - o0[i];
                        w[i] = (c1 - o1[i]) - d0[i];
                    }
                    const R a = w[0] * w[0] + w[1] * w[1] + w[2] * w[2];
                    const R b = d0[0] * w[0] + d0[1] * w[1] + d0[2] * w[2];
                    R u = a > R(0) ? -b / a : R(0);
                    u = u < R(0) ? R(0) : (u > R(1) ? R(1) : u);
                    R d2 = R(0);
                    for (int i = 0; i < 3; ++i) {
                        const R x = d0[i] + u * w[i];
                        d2 += x * x;
                    }
                    const R rr = sph[4 * sp + 3] + ro;
                    hit = hit || (d2 < rr * rr);
                    if (CLEAR) {
                        const R cl = rsqrt_r(d2) - rr;
                        clr = cl < clr ? cl : clr;
                    }
                }
                pairs_total += (unsigned long long)G.S;
                t0 = t1;
            }
        }
        E.hit[e] = hit ? 1 : 0;
        if (CLEAR) atomic_min_r<R>(E.clear + e, clr);  // order-encoded like the discrete path
        ++done;
    }
    const int lane = threadIdx.x & 31;
    if (E.points_done) {
        for (int o = 16; o > 0; o >>= 1) done += __shfl_xor_sync(0xffffffffu, done, o);
        if (lane == 0 && done) atomicAdd(E.points_done, done);
    }
    if (E.pairs_done) {
        for (int o = 16; o > 0; o >>= 1) pairs_total += __shfl_xor_sync(0xffffffffu, pairs_total, o);
        if (lane == 0 && pairs_total) atomicAdd(E.pairs_done, pairs_total);
    }
}

template <typename R>
cudaError_t launch_validate_cont(const Geom<R>& g, const EdgeBatch<R>& e, bool clearance, cudaStream_t st) {
    const int blocks = validate_grid_blocks() * 2;
    if (clearance) k_validate_cont<R, true><<<blocks, 256, 0, st>>>(g, e);
    else k_validate_cont<R, false><<<blocks, 256, 0, st>>>(g, e);
    return cudaGetLastError();
}

// Check-point counts, c = max(1, ceil(max(D, v_max |dt|) / res - 1e-3)),
// evaluated in double from the stored endpoints.
template <typename R>
__global__ void k_edge_counts(double vmax, int dof, const R* qa, const R* ta, const R* qb, const R* tb, int qstride,
                              int n, double res, int* cnt) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    double s2 = 0.0;
    for (int i = 0; i < dof; ++i) {
        double dd = (double)qb[(size_t)e * qstride + i] - (double)qa[(size_t)e * qstride + i];
        s2 = __dadd_rn(s2, __dmul_rn(dd, dd));
    }
    double D = sqrt(s2);
    double L = fmax(D, __dmul_rn(vmax, fabs((double)tb[e] - (double)ta[e])));
    double c = ceil(L / res - 1e-3);
    cnt[e] = c < 1.0 ? 1 : (int)c;
}

template <typename R>
cudaError_t launch_edge_counts(const Geom<R>& g, const R* qa, const R* ta, const R* qb, const R* tb, int qstride,
                               int n, double res, int* cnt, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_edge_counts<R><<<(n + 255) / 256, 256, 0, st>>>(g.vmax_d, g.dof, qa, ta, qb, tb, qstride, n, res, cnt);
    return cudaGetLastError();
}

// Exclusive prefix sum of counts into off[0..n] (off[n] = total); three phases.
constexpr int kScanBlock = 1024;
constexpr int kScanPer = 4;
constexpr int kScanTile = kScanBlock * kScanPer;

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long* sh, long long* total) {
    // Warp scan then scan of warp totals.
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sh[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int nw = blockDim.x >> 5;
        long long w = lane < nw ? sh[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            long long y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        if (lane < nw) sh[lane] = w;
    }
    __syncthreads();
    long long before = (warp > 0 ? sh[warp - 1] : 0) + x - v;
    if (total) *total = sh[(blockDim.x >> 5) - 1];
    __syncthreads();
    return before;
}

__global__ void k_scan_tiles(const int* cnt, int n, long long* off, long long* tile_tot) {
    __shared__ long long sh[32];
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanPer;
    long long v[kScanPer];
    long long sum = 0;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        v[i] = (base + i < n) ? cnt[base + i] : 0;
        sum += v[i];
    }
    long long tot;
    long long pre = block_exclusive_scan(sum, sh, &tot);
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
        if (base + i < n) off[base + i] = pre;
        pre += v[i];
    }
    if (threadIdx.x == 0) tile_tot[blockIdx.x] = tot;
}

__global__ void k_scan_tops(long long* tile_tot, int ntiles, long long* off, int n) {
    __shared__ long long sh[32];
    long long carry = 0;
    for (int b0 = 0; b0 < ntiles; b0 += blockDim.x) {
        int b = b0 + threadIdx.x;
        long long v = b < ntiles ? tile_tot[b] : 0;
        long long tot;
        long long pre = block_exclusive_scan(v, sh, &tot);
        if (b < ntiles) tile_tot[b] = carry + pre;
        carry += tot;
    }
    if (threadIdx.x == 0) off[n] = carry;
}

__global__ void k_scan_add(long long* off, int n, const long long* tile_tot) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) off[i] += tile_tot[i / kScanTile];
}

cudaError_t launch_scan_counts(const int* cnt, int n, long long* off, long long* tile_tmp, cudaStream_t st) {
    if (n <= 0) {
        return cudaMemsetAsync(off, 0, sizeof(long long), st);
    }
    int ntiles = (n + kScanTile - 1) / kScanTile;
    k_scan_tiles<<<ntiles, kScanBlock, 0, st>>>(cnt, n, off, tile_tmp);
    k_scan_tops<<<1, kScanBlock, 0, st>>>(tile_tmp, ntiles, off, n);
    k_scan_add<<<(n + 255) / 256, 256, 0, st>>>(off, n, tile_tmp);
    return cudaGetLastError();
}

// Small fills and conversions used by the batch entry point.
__global__ void k_fill_u32(unsigned* p, long long n, unsigned v) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}
__global__ void k_fill_u64(unsigned long long* p, long long n, unsigned long long v) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}
cudaError_t launch_fill(void* p, long long n, int bytes, unsigned long long v, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    int grid = (int)((n + 255) / 256);
    if (bytes == 4) k_fill_u32<<<grid, 256, 0, st>>>((unsigned*)p, n, (unsigned)v);
    else k_fill_u64<<<grid, 256, 0, st>>>((unsigned long long*)p, n, v);
    return cudaGetLastError();
}

template <typename R>
__global__ void k_finish_batch(int n, const int* hit, unsigned char* verdict, R* clear) {
    int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n) return;
    verdict[e] = hit[e] ? 0 : 1;
    if (clear) clear[e] = ord_dec(*reinterpret_cast<const decltype(ord_enc(R(0)))*>(clear + e));
}
template <typename R>
cudaError_t launch_finish_batch(int n, const int* hit, unsigned char* verdict, R* clear, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_finish_batch<R><<<(n + 255) / 256, 256, 0, st>>>(n, hit, verdict, clear);
    return cudaGetLastError();
}
template cudaError_t launch_finish_batch<float>(int, const int*, unsigned char*, float*, cudaStream_t);
template cudaError_t launch_finish_batch<double>(int, const int*, unsigned char*, double*, cudaStream_t);

template cudaError_t launch_validate<float>(const Geom<float>&, const Geom<float>&, const EdgeBatch<float>&, bool, bool,
                                            cudaStream_t);
template cudaError_t launch_validate<double>(const Geom<double>&, const Geom<float>&, const EdgeBatch<double>&, bool,
                                             bool, cudaStream_t);
template cudaError_t launch_validate_full<float>(const Geom<float>&, const EdgeBatch<float>&, bool, cudaStream_t);
template cudaError_t launch_validate_full<double>(const Geom<double>&, const EdgeBatch<double>&, bool, cudaStream_t);
template cudaError_t launch_validate_cont<float>(const Geom<float>&, const EdgeBatch<float>&, bool, cudaStream_t);
template cudaError_t launch_validate_cont<double>(const Geom<double>&, const EdgeBatch<double>&, bool, cudaStream_t);
template cudaError_t launch_edge_counts<float>(const Geom<float>&, const float*, const float*, const float*,
                                               const float*, int, int, double, int*, cudaStream_t);
template cudaError_t launch_edge_counts<double>(const Geom<double>&, const double*, const double*, const double*,
                                                const double*, int, int, double, int*, cudaStream_t);

}  // namespace stp
