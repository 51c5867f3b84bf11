// Allocation-free ForceAtlas2 iteration on caller-owned device arrays.
//
// Some callers cannot call cudaMalloc at the point where they want to run a
// layout step: a serving process that hands all of its device memory to
// its own pool at start-up has nothing left for a library to allocate, and
// a latency-bound loop cannot afford the device-wide synchronisation that
// cudaMalloc and cudaFree may cause.  bgl_fa2_iteration_noalloc serves them:
// the caller passes every input and output, and the only scratch the
// iteration needs -- above eight tiles the per-tile swing/traction partial
// sums and the arrival counter of their reduction -- lives in one file-scope device
// array of fixed size (NOALLOC_SCRATCH_BYTES), which every GPU that loads
// this library holds until the process exits.
//
// The kernels are variants of the ones in fa2.cu that need no host-built
// tile list and no per-call buffers: one component, targets tiled by block
// index, the stages of a tile's sources spread over a thread-block cluster
// whose blocks hand their sums over in distributed shared memory, or, on large
// components, all in one block.  The
// formulas of every force term, of the swing/traction sums and of the update
// are the same; the order and precision of the sums differ (here every thread
// sums its swing/traction terms in FP64 over tiles of 2,048 nodes and a hub's
// attraction is summed entry after entry, where fa2.cu sums in FP32 within a
// warp over tiles of 256 nodes and splits hub rows into 2,048-entry chunks),
// so the two agree within rounding, not bitwise.  A position that becomes
// non-finite sets the context's d_flag[2], which bgl_ctx_sync reports.
#include <algorithm>

#include <cooperative_groups.h>

#include "bgl_internal.cuh"
#include "p2p.cuh"

namespace bgl {

namespace {

namespace cg = cooperative_groups;

constexpr int NA_TILE = 128;                      // targets per cluster, one a thread
constexpr int NA_CLUSTER = 8;                     // blocks per cluster (the portable maximum)
constexpr int NA_STILE = 1024;                    // sources per shared-memory stage
constexpr int NA_LANE_DEG = 8;                    // nodes up to this degree: attraction by one lane
constexpr int NA_RED_TILE = 2048;                 // nodes per swing/traction tile
constexpr int64_t NA_MAX_NODES = BGL_NOALLOC_MAX_NODES;
constexpr int NA_MAX_TILES = (int)(NA_MAX_NODES / NA_RED_TILE);
constexpr size_t NA_COUNTER_BYTES = 256;          // arrival counter, padded
constexpr size_t NOALLOC_SCRATCH_BYTES = NA_COUNTER_BYTES + sizeof(double2) * NA_MAX_TILES;

// The scratch of every call on this device: [0, 256) the arrival counter,
// then NA_MAX_TILES double2 partial sums.  Host code must not pass this
// symbol to a kernel; it passes the device address from
// cudaGetSymbolAddress (noalloc_scratch_address, stored in the context).
static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_SCRATCH_BYTES];

// NA_STILE sources from s0 on (cnt of them) to src, by a block of NA_TILE
__device__ __forceinline__ void na_stage(const float2 *__restrict__ xy, const float *__restrict__ mass, int64_t s0,
                                         int cnt, float4 *src) {
#pragma unroll
    for (int k = 0; k < NA_STILE / NA_TILE; ++k) {
        const int j = k * NA_TILE + threadIdx.x;
        if (j < cnt) {
            const float2 p = xy[s0 + j];
            src[j] = make_float4(p.x, p.y, mass[s0 + j], 0.f);
        }
    }
}

// A stage's sum v enters the compensated running total s (c: the rounding so far)
__device__ __forceinline__ void na_add(float v, float &s, float &c) {
    const float y = v - c, t = s + y;
    c = (t - s) - y;
    s = t;
}

// F of a node at z from its repulsion sum and attraction (the repulsion rounded before the attraction)
__device__ __forceinline__ float2 na_total(float m, float kr, float kg, float sx, float sy, float2 a, float2 z) {
    const float km = kr * m, kgm = kg * m;
    const float2 fr = make_float2(__fmul_rn(km, sx), __fmul_rn(km, sy));
    return make_float2((fr.x + a.x) - kgm * z.x, (fr.y + a.y) - kgm * z.y);
}

// Forces of the cluster's NA_TILE targets: repulsion from all n nodes, plus
// attraction and gravity.
//
// A target's repulsion is a chain over its sources (each 1,024-source stage's
// sum enters a compensated total), so the cluster's blocks take the stages in
// turn; block 0 adds their sums in order out of the others' shared memory
// (two buffers, so one barrier a round).  A cluster has a block per stage and
// one more, up to NA_CLUSTER: on a small component more would only share SMs
// with the ones that work.  The blocks without a stage, or all of them,
// share the attraction, entry after entry: a lane for a node of few entries,
// for the others the warp loads 32 entries at a time and adds them in order
// through shuffles.  No memory is needed beyond the blocks' own.  One block
// per 512 targets with all stages, and a kernel with one thread per node for
// the attraction, took 99.6 and 15.5 us for 2,821 nodes.
__global__ void __launch_bounds__(NA_TILE)
    na_force_kernel(const float2 *__restrict__ xy, const float *__restrict__ mass, const int64_t *__restrict__ off,
                    const int32_t *__restrict__ adj, int64_t n, float kr, float kg, float2 *__restrict__ f) {
    __shared__ float4 src[NA_STILE + P2P_AHEAD];
    __shared__ float2 part[2][NA_TILE];
    __shared__ float2 satt[NA_TILE];
    const cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), blocks = (int)cluster.num_blocks();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t0 = (int64_t)(blockIdx.x / (unsigned)blocks) * NA_TILE;
    const int64_t stages = (n + NA_STILE - 1) / NA_STILE;
    // attraction: shared by the blocks without a stage, or by all of them
    const int first = stages < blocks ? (int)stages : 0;
    const int share = (NA_TILE + blocks - first - 1) / (blocks - first);
    if (rank >= first) {
        const int per_warp = (share + NA_TILE / 32 - 1) / (NA_TILE / 32);
        const int node = warp * per_warp + lane;         // lanes below per_warp own a node
        const int i = (rank - first) * share + node;
        const int64_t q = t0 + i;
        const bool own = lane < per_warp && node < share && i < NA_TILE, ok = own && q < n;
        const int64_t e0 = ok ? off[q] : 0, deg = ok ? off[q + 1] - e0 : 0;
        const float2 p = ok ? xy[q] : make_float2(0.f, 0.f);
        float ax = 0.f, ay = 0.f;
        if (deg <= NA_LANE_DEG) {
            float2 o[NA_LANE_DEG];
#pragma unroll
            for (int e = 0; e < NA_LANE_DEG; ++e) o[e] = e < deg ? xy[adj[e0 + e]] : p;
#pragma unroll
            for (int e = 0; e < NA_LANE_DEG; ++e) {
                if (e < deg) {
                    ax -= p.x - o[e].x;
                    ay -= p.y - o[e].y;
                }
            }
        }
        unsigned more = __ballot_sync(0xffffffffu, deg > NA_LANE_DEG);
        while (more) {
            const int l = __ffs(more) - 1;
            more &= more - 1;
            const int64_t f0 = __shfl_sync(0xffffffffu, e0, l), d = __shfl_sync(0xffffffffu, deg, l);
            const float px = __shfl_sync(0xffffffffu, p.x, l), py = __shfl_sync(0xffffffffu, p.y, l);
            float sx = 0.f, sy = 0.f;
            constexpr int C = 4;                         // loads of four rounds in flight
            for (int64_t c0 = 0; c0 < d; c0 += 32 * C) {
                float2 t[C];
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int64_t e = c0 + c * 32 + lane;
                    const float2 o = e < d ? xy[adj[f0 + e]] : make_float2(px, py);
                    t[c] = make_float2(px - o.x, py - o.y);
                }
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const int m = (int)min((int64_t)32, d - c0 - c * 32);
#pragma unroll 8
                    for (int j = 0; j < m; ++j) {
                        sx -= __shfl_sync(0xffffffffu, t[c].x, j);
                        sy -= __shfl_sync(0xffffffffu, t[c].y, j);
                    }
                }
            }
            if (lane == l) {
                ax = sx;
                ay = sy;
            }
        }
        if (own) satt[node] = make_float2(ax, ay);
    }
    const int64_t q = t0 + threadIdx.x;
    const float2 z = q < n ? xy[q] : make_float2(0.f, 0.f);
    float sx = 0.f, sy = 0.f, cx = 0.f, cy = 0.f;        // block 0: the running total
    int buf = 0;
    for (int64_t k0 = 0; k0 < stages; k0 += blocks, buf ^= 1) {
        const int64_t s0 = (k0 + rank) * NA_STILE;
        const int cnt = (int)(s0 >= n ? 0 : (n - s0 < NA_STILE ? n - s0 : NA_STILE));
        __syncthreads();
        na_stage(xy, mass, s0, cnt, src);
        __syncthreads();
        float ax = 0.f, ay = 0.f;
        // (the node itself adds 0)
        p2p_chain(z.x, z.y, src, cnt, [](float dx, float dy) { return fmaxf(fmaf(dx, dx, dy * dy), 1e-30f); }, ax, ay);
        part[buf][threadIdx.x] = make_float2(ax, ay);
        cluster.sync();
        if (rank == 0) {
            const int m = (int)(stages - k0 < blocks ? stages - k0 : blocks);
            for (int r = 0; r < m; ++r) {                // compensated running total of the stage sums
                const float2 v = cluster.map_shared_rank(&part[0][0], r)[buf * NA_TILE + threadIdx.x];
                na_add(v.x, sx, cx);
                na_add(v.y, sy, cy);
            }
        }
    }
    if (rank == 0 && q < n) {
        const float2 a = cluster.map_shared_rank(&satt[0], first + threadIdx.x / share)[threadIdx.x % share];
        f[q] = na_total(mass[q], kr, kg, sx, sy, a, z);
    }
    cluster.sync();                                      // no block leaves while block 0 reads its memory
}

// Attraction of the warp's nodes q, a lane each (ok: the lane has one), in
// the order and the manner of na_force_kernel, which has it written out: with
// a call of this it ran 3 % slower, at two registers less.
__device__ __forceinline__ float2 na_attraction(const float2 *__restrict__ xy, const int64_t *__restrict__ off,
                                                const int32_t *__restrict__ adj, int64_t q, bool ok) {
    const int lane = threadIdx.x & 31;
    const int64_t e0 = ok ? off[q] : 0, deg = ok ? off[q + 1] - e0 : 0;
    const float2 p = ok ? xy[q] : make_float2(0.f, 0.f);
    float ax = 0.f, ay = 0.f;
    if (deg <= NA_LANE_DEG) {
        float2 o[NA_LANE_DEG];
#pragma unroll
        for (int e = 0; e < NA_LANE_DEG; ++e) o[e] = e < deg ? xy[adj[e0 + e]] : p;
#pragma unroll
        for (int e = 0; e < NA_LANE_DEG; ++e) {
            if (e < deg) {
                ax -= p.x - o[e].x;
                ay -= p.y - o[e].y;
            }
        }
    }
    unsigned more = __ballot_sync(0xffffffffu, deg > NA_LANE_DEG);
    while (more) {
        const int l = __ffs(more) - 1;
        more &= more - 1;
        const int64_t f0 = __shfl_sync(0xffffffffu, e0, l), d = __shfl_sync(0xffffffffu, deg, l);
        const float px = __shfl_sync(0xffffffffu, p.x, l), py = __shfl_sync(0xffffffffu, p.y, l);
        float sx = 0.f, sy = 0.f;
        constexpr int C = 4;                             // loads of four rounds in flight
        for (int64_t c0 = 0; c0 < d; c0 += 32 * C) {
            float2 t[C];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int64_t e = c0 + c * 32 + lane;
                const float2 o = e < d ? xy[adj[f0 + e]] : make_float2(px, py);
                t[c] = make_float2(px - o.x, py - o.y);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int m = (int)min((int64_t)32, d - c0 - c * 32);
#pragma unroll 8
                for (int j = 0; j < m; ++j) {
                    sx -= __shfl_sync(0xffffffffu, t[c].x, j);
                    sy -= __shfl_sync(0xffffffffu, t[c].y, j);
                }
            }
        }
        if (lane == l) {
            ax = sx;
            ay = sy;
        }
    }
    return make_float2(ax, ay);
}

// The same for a component with targets enough to fill the chip without a
// split of the stages: a block has 2 NA_TILE targets, two a thread in packed
// FP32x2 arithmetic, and all stages, so that a source is read from shared
// memory once for two pairs and no block waits for another.  Bound by issue and
// the MUFU; the sums are the cluster kernel's bit for bit.  The line lies where
// the blocks are some seven an SM: on 131,072 nodes 5.73 ms an iteration with
// the clusters and 5.97 with this, on 196,608 12.8 and 12.9, on 262,144 22.8
// and 19.8, on 1,048,576 363 and 270 (two scalar targets a thread in blocks
// of 512, with the attraction in a kernel of its own: 339).
constexpr int64_t NA_WIDE_MIN = 1 << 18;

__global__ void __launch_bounds__(NA_TILE)
    na_force_wide_kernel(const float2 *__restrict__ xy, const float *__restrict__ mass,
                         const int64_t *__restrict__ off, const int32_t *__restrict__ adj, int64_t n, float kr,
                         float kg, float2 *__restrict__ f) {
    __shared__ float4 src[NA_STILE];
    const int64_t q0 = (int64_t)blockIdx.x * (2 * NA_TILE) + threadIdx.x;
    float2 z[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) z[r] = q0 + r * NA_TILE < n ? xy[q0 + r * NA_TILE] : make_float2(0.f, 0.f);
    // negated targets and sums: each operation is the sign mirror of p2p_chain's
    const float2 nzx = make_float2(-z[0].x, -z[1].x), nzy = make_float2(-z[0].y, -z[1].y);
    float sx[2] = {0.f, 0.f}, sy[2] = {0.f, 0.f}, cx[2] = {0.f, 0.f}, cy[2] = {0.f, 0.f};
    for (int64_t s0 = 0; s0 < n; s0 += NA_STILE) {
        const int cnt = (int)(n - s0 < NA_STILE ? n - s0 : NA_STILE);
        __syncthreads();
        na_stage(xy, mass, s0, cnt, src);
        __syncthreads();
        float2 gx = make_float2(0.f, 0.f), gy = make_float2(0.f, 0.f);
#pragma unroll 4
        for (int j = 0; j < cnt; ++j) {
            const float4 q = src[j];
            const float2 dx = __fadd2_rn(make_float2(q.x, q.x), nzx), dy = __fadd2_rn(make_float2(q.y, q.y), nzy);
            const float2 r2 = __ffma2_rn(dx, dx, __fmul2_rn(dy, dy));
            const float2 inv = make_float2(rcp_approx(fmaxf(r2.x, 1e-30f)), rcp_approx(fmaxf(r2.y, 1e-30f)));
            const float2 w = __fmul2_rn(make_float2(q.z, q.z), inv);
            gx = __ffma2_rn(w, dx, gx);
            gy = __ffma2_rn(w, dy, gy);
        }
        na_add(-gx.x, sx[0], cx[0]);
        na_add(-gx.y, sx[1], cx[1]);
        na_add(-gy.x, sy[0], cy[0]);
        na_add(-gy.y, sy[1], cy[1]);
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int64_t q = q0 + r * NA_TILE;
        const float2 a = na_attraction(xy, off, adj, q, q < n);
        if (q < n) f[q] = na_total(mass[q], kr, kg, sx[r], sy[r], a, z[r]);
    }
}

// Swing and traction sums of the nodes of the block's tile (256 threads; the
// result in thread 0): each thread's terms in order, lanes by an exchange
// sum, warps in order.  F and P are the thread's forces and previous forces.
constexpr int NA_PER = NA_RED_TILE / 256;
__device__ __forceinline__ double2 na_tile_sums(const float2 (&F)[NA_PER], const float2 (&P)[NA_PER],
                                                const float (&m)[NA_PER], int64_t q0, int64_t t1, int variant) {
    __shared__ double ws[32], wt[32];
    double sw = 0.0, tr = 0.0;
#pragma unroll
    for (int k = 0; k < NA_PER; ++k) {
        if (q0 + k * 256 >= t1) break;
        const float s = sqrtf((F[k].x - P[k].x) * (F[k].x - P[k].x) + (F[k].y - P[k].y) * (F[k].y - P[k].y));
        const float u = sqrtf((F[k].x + P[k].x) * (F[k].x + P[k].x) + (F[k].y + P[k].y) * (F[k].y + P[k].y));
        if (variant == 1) {
            sw += (double)m[k] * s;
            tr += 0.5 * (double)m[k] * u;
        } else {
            sw += s;
            tr += u;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sw += __shfl_xor_sync(0xffffffffu, sw, o);
        tr += __shfl_xor_sync(0xffffffffu, tr, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        ws[warp] = sw;
        wt[warp] = tr;
    }
    __syncthreads();
    double s = 0.0, u = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            s += ws[w];
            u += wt[w];
        }
    return make_double2(s, u);
}

// s_G = min(tau trc / swg, 1.5 s_G)
__device__ __forceinline__ double na_speed(double swg, double trc, double g, double tau) {
    double s_new = swg > 0.0 ? tau * trc / swg : 1.5 * g;
    if (s_new > 1.5 * g) s_new = 1.5 * g;
    return s_new;
}

// the node's move at global speed g
__device__ __forceinline__ float2 na_move(float2 p, float2 F, float2 P, float g, float ks, float ksmax, int *bad) {
    float sw = sqrtf((F.x - P.x) * (F.x - P.x) + (F.y - P.y) * (F.y - P.y));
    float s = ks * g / (1.f + g * sqrtf(sw));
    float fn = sqrtf(F.x * F.x + F.y * F.y);
    if (fn > 0.f && s > ksmax / fn) s = ksmax / fn;
    p.x += s * F.x;
    p.y += s * F.y;
    if (!isfinite(p.x) || !isfinite(p.y)) *bad = 1;
    return p;
}

// Swing, traction, global speed and update of a component of up to NA_CLUSTER
// tiles in one kernel: a cluster with a block per tile, the tiles' sums read
// through distributed shared memory and added in tile order by every block.
// Each node's forces are read once.  The sums and the update as two kernels
// are all latency at this size (8.6 + 3.5 us and a launch between them at
// 2,821 nodes): a whole iteration on 2,821 nodes 29.0 us with two kernels and
// 27.9 with this one, on 8,192 48.5 and 46.6, on 16,384 (eight tiles, the most
// a cluster holds) 124.6 and 122.8.
__global__ void __launch_bounds__(256) na_swing_update_kernel(const float2 *__restrict__ f, float2 *__restrict__ fprev,
                                                              const float *__restrict__ mass,
                                                              float2 *__restrict__ xy, int64_t n, int variant,
                                                              double tau, double *sg, float ks, float ksmax,
                                                              int *bad) {
    __shared__ double2 tile;
    const cg::cluster_group cluster = cg::this_cluster();
    const int64_t t0 = (int64_t)blockIdx.x * NA_RED_TILE;
    const int64_t t1 = t0 + NA_RED_TILE < n ? t0 + NA_RED_TILE : n;
    const int64_t q0 = t0 + threadIdx.x;
    float2 F[NA_PER], P[NA_PER], p[NA_PER];
    float m[NA_PER];
#pragma unroll
    for (int k = 0; k < NA_PER; ++k) {
        const int64_t q = q0 + k * 256;
        F[k] = q < t1 ? f[q] : make_float2(0.f, 0.f);
        P[k] = q < t1 ? fprev[q] : make_float2(0.f, 0.f);
        m[k] = variant == 1 && q < t1 ? mass[q] : 0.f;
        p[k] = q < t1 ? xy[q] : make_float2(0.f, 0.f);
    }
    const double g0 = *sg;
    const double2 own = na_tile_sums(F, P, m, q0, t1, variant);
    if (threadIdx.x == 0) tile = own;
    cluster.sync();                        // the tiles' sums; every thread has read *sg
    double swg = 0.0, trc = 0.0;
    for (unsigned k = 0; k < gridDim.x; ++k) {
        const double2 v = *cluster.map_shared_rank(&tile, k);
        swg += v.x;
        trc += v.y;
    }
    const double s_new = na_speed(swg, trc, g0, tau);
    if (blockIdx.x == 0 && threadIdx.x == 0) *sg = s_new;
    const float g = (float)s_new;
#pragma unroll
    for (int k = 0; k < NA_PER; ++k) {
        const int64_t q = q0 + k * 256;
        if (q >= t1) break;
        xy[q] = na_move(p[k], F[k], P[k], g, ks, ksmax, bad);
        fprev[q] = F[k];
    }
    cluster.sync();                        // no block leaves while another reads its sum
}

// Larger components: partial sums per tile into the static scratch; the last
// block sums the tiles in order and sets s_G
__global__ void na_swing_traction_kernel(const float2 *__restrict__ f, const float2 *__restrict__ fprev,
                                         const float *__restrict__ mass, int64_t n, int variant, double tau,
                                         double *sg, unsigned char *scratch) {
    __shared__ bool last;
    unsigned *counter = reinterpret_cast<unsigned *>(scratch);
    double2 *partial = reinterpret_cast<double2 *>(scratch + NA_COUNTER_BYTES);
    const int64_t t0 = (int64_t)blockIdx.x * NA_RED_TILE;
    const int64_t t1 = t0 + NA_RED_TILE < n ? t0 + NA_RED_TILE : n;
    // the tile's loads in flight together, then each thread's terms in order
    float2 F[NA_PER], P[NA_PER];
    float m[NA_PER];
#pragma unroll
    for (int k = 0; k < NA_PER; ++k) {
        const int64_t q = t0 + k * 256 + threadIdx.x;
        F[k] = q < t1 ? f[q] : make_float2(0.f, 0.f);
        P[k] = q < t1 ? fprev[q] : make_float2(0.f, 0.f);
        m[k] = variant == 1 && q < t1 ? mass[q] : 0.f;
    }
    const double2 own = na_tile_sums(F, P, m, t0 + threadIdx.x, t1, variant);
    if (threadIdx.x == 0) {
        partial[blockIdx.x] = own;
        __threadfence();
        last = atomicAdd(counter, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // the tiles' sums fetched together, then added in order
    __shared__ double2 tiles[NA_MAX_TILES];
    for (unsigned k = threadIdx.x; k < gridDim.x; k += blockDim.x) tiles[k] = __ldcg(&partial[k]);
    __syncthreads();
    if (threadIdx.x != 0) return;
    double swg = 0.0, trc = 0.0;
    for (unsigned k = 0; k < gridDim.x; ++k) {
        swg += tiles[k].x;
        trc += tiles[k].y;
    }
    *sg = na_speed(swg, trc, *sg, tau);
    *counter = 0u;
}

__global__ void na_update_kernel(const float2 *__restrict__ f, float2 *__restrict__ fprev, float2 *__restrict__ xy,
                                 const double *__restrict__ sg, int64_t n, float ks, float ksmax, int *bad,
                                 unsigned char *scratch) {
    // the arrival counter of the next call starts at zero whatever ran before
    if (blockIdx.x == 0 && threadIdx.x == 0) *reinterpret_cast<unsigned *>(scratch) = 0u;
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const float2 F = f[q];
    xy[q] = na_move(xy[q], F, fprev[q], (float)*sg, ks, ksmax, bad);
    fprev[q] = F;
}

inline unsigned na_blocks(int64_t n, int64_t per) { return (unsigned)((n + per - 1) / per); }

}  // namespace

// Device address of the scratch array on the current device.  Called by
// bgl_ctx_create with the context's device current, so every context holds
// the address for its device (a context created after a device reset looks
// it up again).
void *noalloc_scratch_address() {
    void *ptr = nullptr;
    BGL_CUDA(cudaGetSymbolAddress(&ptr, g_noalloc_scratch));
    return ptr;
}

void fa2_iteration_noalloc(bgl_ctx *c, int64_t n, const int64_t *d_off, const int32_t *d_adj, const float *d_mass,
                           float2 *d_xy, float2 *d_fprev, float2 *d_f, double *d_sg, const bgl_params *p) {
    BGL_REQUIRE(n >= 0, "noalloc: n must be >= 0");
    BGL_REQUIRE(n <= NA_MAX_NODES, "noalloc: component has more than BGL_NOALLOC_MAX_NODES (2^20) nodes");
    if (n == 0) return;
    BGL_REQUIRE(d_off && d_adj && d_mass && d_xy && d_fprev && d_f && d_sg, "noalloc: a device array is NULL");
    unsigned char *scratch = c->noalloc_scratch;
    BGL_REQUIRE(scratch != nullptr, "noalloc: the context has no scratch address");
    cudaStream_t s = c->stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    if (n < NA_WIDE_MIN) {
        attr.val.clusterDim.x = (unsigned)std::min<int64_t>(NA_CLUSTER, (n + NA_STILE - 1) / NA_STILE + 1);
        cfg.gridDim = dim3(na_blocks(n, NA_TILE) * attr.val.clusterDim.x);
        cfg.blockDim = dim3(NA_TILE);
        BGL_CUDA(cudaLaunchKernelEx(&cfg, na_force_kernel, (const float2 *)d_xy, d_mass, d_off, d_adj, n,
                                    (float)p->kr, (float)p->kg, d_f));
        BGL_LAUNCH_CHECK();
    } else {
        na_force_wide_kernel<<<na_blocks(n, 2 * NA_TILE), NA_TILE, 0, s>>>(d_xy, d_mass, d_off, d_adj, n,
                                                                          (float)p->kr, (float)p->kg, d_f);
        BGL_LAUNCH_CHECK();
    }
    const unsigned tiles = na_blocks(n, NA_RED_TILE);
    if (tiles <= NA_CLUSTER) {
        attr.val.clusterDim.x = tiles;
        cfg.gridDim = dim3(tiles);
        cfg.blockDim = dim3(256);
        BGL_CUDA(cudaLaunchKernelEx(&cfg, na_swing_update_kernel, (const float2 *)d_f, d_fprev, d_mass, d_xy, n,
                                    (int)p->swing_variant, p->tau, d_sg, (float)p->ks, (float)p->ksmax,
                                    c->d_flag + 2));
        BGL_LAUNCH_CHECK();
        return;
    }
    na_swing_traction_kernel<<<tiles, 256, 0, s>>>(d_f, d_fprev, d_mass, n, p->swing_variant,
                                                                       p->tau, d_sg, scratch);
    BGL_LAUNCH_CHECK();
    na_update_kernel<<<na_blocks(n, 256), 256, 0, s>>>(d_f, d_fprev, d_xy, d_sg, n, (float)p->ks, (float)p->ksmax,
                                                       c->d_flag + 2, scratch);
    BGL_LAUNCH_CHECK();
}

}  // namespace bgl
