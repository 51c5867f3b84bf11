// ForceAtlas2 iteration (Section 3.2) on the device.
//
// One iteration over the ForceAtlas2 components [c0, c1):
//   K1 repulsion      f <- F_rep = kr m_i sum_j m_j (p_i - p_j) / |p_i - p_j|^2.
//                     Exact components: exact_kernel, a block per tile of 128
//                     or 256 targets and stage of 1,024 sources, or per tile
//                     with all sources (ExactSum).  FMM components: fmm.cu.
//   K2 attraction     -sum_{j adjacent} (p_i - p_j) - kg m_i p_i, added to f.
//      + gravity      Exact: blocks of their own in exact_kernel's launch;
//                     the tile's last block to finish adds what they sum.
//                     FMM: attraction_gravity_kernel on a second stream beside
//                     the evaluation, whose final kernel adds fa.  Nodes of
//                     degree > 128 in chunks of 2,048 entries, in chunk order
//   K3 swing/traction |F_t - F_{t-1}|, |F_t + F_{t-1}| summed in FP32 over 32
//                     nodes and in FP64 above (SwingArgs); a component's last
//                     block to finish sets s_G = min(tau trc / swg, 1.5 s_G).
//                     Exact: in exact_kernel.  FMM: in combine_kernel (fmm.cu)
//                     for a component that runs alone, else
//                     swing_traction_kernel
//   K4 update         s_n = ks s_G / (1 + s_G sqrt|F_t - F_{t-1}|), capped at
//                     ksmax / |F_t|; p_n += s_n F_t; F_{t-1} <- F_t
//                     (update_kernel; with the next root square in
//                     update_root_kernel, fmm.cu, for an FMM component alone)
// The sequence has fixed launch shapes, so a few iterations are captured as
// the body of a device-side WHILE loop in a CUDA graph: one launch runs them
// all.  Every sum has a fixed order, so runs are bitwise reproducible.
#include <algorithm>
#include <cstdlib>
#include <cstring>

#include "bgl_internal.cuh"
#include "fa2_update.cuh"
#include "fmm.cuh"
#include "p2p.cuh"

namespace bgl {

namespace {

constexpr int EX_THREADS = 128, EX_WARPS = EX_THREADS / 32;
constexpr int EX_STAGE = 1024;                 // sources summed before they enter the compensated total
constexpr int64_t EX_SPLIT_MAX_N = 1 << 16;    // components up to this size: a block per stage (partial sums in memory)
// Partial sums take 8 bytes a node and stage: up to 64 a node for components
// of up to EX_SPLIT_FREE_N nodes, 512 on 65,536.  All components above
// EX_SPLIT_FREE_N of a run together get EX_PART_BYTES, smallest first: sixteen
// of 65,536.  More have tiles enough to fill the chip without a split (of
// 60,000 nodes, times of some iterations split and not: 3 components 24.6 and
// 34.1 ms, 10 33.5 and 34.6, 16 52.9 and 52.9, 30 52.5 and 48.8, the last with
// 875 MB of partial sums).
constexpr int64_t EX_SPLIT_FREE_N = 8 * EX_STAGE;
constexpr int64_t EX_PART_BYTES = int64_t(512) << 20;
#ifndef BGL_EXACT_WIDE_WARPS
#define BGL_EXACT_WIDE_WARPS 3000              // warps at two targets per lane from which a run takes two
#endif
constexpr int ATT_LANE_DEG = 8;                // attraction: nodes up to this degree by one lane each
constexpr int HEAVY_DEG = 128;
constexpr int HEAVY_CHUNK = 2048;              // adjacency entries per block for high-degree nodes
constexpr int RED_TILE = 256;                  // nodes per swing/traction tile (one per thread)

struct Tile {
    int32_t comp;      // component index relative to c0
    int32_t pad;
    int64_t t0, t1;    // target positions [t0, t1)
};


// Swing and traction sums of a component (Section 3.2).  One order for
// every kernel that makes them (here and the fused FMM iteration's
// combine_kernel), so that a component gets the same s_G whatever runs it:
// FP32 over 32 consecutive nodes (a butterfly), FP64 over the eight such
// groups of a 256-node tile, then thread t of 256 over the tiles t, t + 256,
// ..., a butterfly in each warp, and the warps in order.  (FP64 issue is
// scarce on this part, so it is kept off the per-node path.)
struct SwingArgs {
    const float2 *fprev;      // F_{t-1} (null in the exact kernel: forces only)
    int variant;
    double tau;
    double2 *partial;         // one per 256-node tile (swing_traction_kernel)
    float2 *group;            // one per 32 nodes (exact kernel)
    const int32_t *tile_off;  // per component: its first tile, [ncomp + 1] (equal: no tiles here)
    double *sg;               // [ncomp]
    unsigned *counter;        // [ncomp] tiles of each component done, zero between launches
    double *stats;            // optional, component 0
    int *iter;                // iteration counter for stats
};

// s_G from the component's sums, by one thread of its last block to finish
__device__ __forceinline__ void swing_finish(const SwingArgs &a, int comp, double swg, double trc) {
    const double s_new = fa2_global_speed(swg, trc, a.sg[comp], a.tau);
    a.sg[comp] = s_new;
    if (comp == 0) {
        if (a.stats) {
            const int it = *a.iter;
            a.stats[3 * it] = swg;
            a.stats[3 * it + 1] = trc;
            a.stats[3 * it + 2] = s_new;
        }
        *a.iter += 1;
    }
    a.counter[comp] = 0u;
}

__device__ __forceinline__ void warp_sum2(float &x, float &y) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
}
__device__ __forceinline__ void warp_sum2(double &x, double &y) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        x += __shfl_xor_sync(0xffffffffu, x, o);
        y += __shfl_xor_sync(0xffffffffu, y, o);
    }
}

// One block of the exact sum: EX_THREADS R targets of a component (a tile)
// against one stage of its sources, or against all of them, or the tile's
// attraction and gravity (component-order positions).
struct ExBlock {
    int32_t t0, nt;           // targets [t0, t0 + nt)
    int32_t s0, s1;           // sources [s0, s1) (empty: attraction and gravity)
    int32_t comp, tile;       // component relative to c0, tile index (over all components)
    int32_t k, parts;         // part k of `parts` partial sums of the tile
    int32_t part, n;          // the tile's first partial sum in units of a tile's targets; component size
};

struct ExArgs {
    const ExBlock *blk;
    int first;                // block 0 of the launch (past the attraction blocks: repulsion only)
    bool att;
    const float2 *xy;         // xy[q - qbase]
    const float *mass;        // mass[q]
    const int64_t *coff;
    const int32_t *cadj;
    int64_t qbase, fbase;     // f[q - fbase], fa and fprev likewise
    float kr, kg;
    float2 *part;             // partial sums
    unsigned *arrive;         // [tiles] blocks of the tile done, zero between launches
    float2 *fa;               // attraction and gravity
    float2 *f;
    SwingArgs sw;
};

// Attraction and gravity of a tile: -sum_{j adjacent} (p_i - p_j) - kg m_i p_i,
// in the order of attraction_gravity_kernel (one after another up to
// HEAVY_DEG entries, chunks of HEAVY_CHUNK above).  A lane sums a node of up
// to ATT_LANE_DEG entries; for one of up to HEAVY_DEG the warp loads 32
// entries at a time and adds them in order through shuffles (one thread
// loading them took 10 us for a node of 120); the rest the block takes.
template <int R>
__device__ void tile_attraction(const ExArgs &a, const ExBlock &b) {
    __shared__ float2 hred[8];
    __shared__ int hlist[EX_THREADS * R], nh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float2 *__restrict__ xy = a.xy - a.qbase;
    if (threadIdx.x == 0) nh = 0;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = (warp * R + r) * 32 + lane;
        const int q = b.t0 + i;
        const bool ok = i < b.nt;
        const int64_t e0 = ok ? a.coff[q] : 0, deg = ok ? a.coff[q + 1] - e0 : 0;
        const float2 p = ok ? xy[q] : make_float2(0.f, 0.f);
        float ax = 0.f, ay = 0.f;
        if (deg <= ATT_LANE_DEG) {
            float2 o[ATT_LANE_DEG];
#pragma unroll
            for (int e = 0; e < ATT_LANE_DEG; ++e) o[e] = e < deg ? xy[a.cadj[e0 + e]] : p;
#pragma unroll
            for (int e = 0; e < ATT_LANE_DEG; ++e) {
                if (e < deg) {
                    ax -= p.x - o[e].x;
                    ay -= p.y - o[e].y;
                }
            }
        }
        if (deg > HEAVY_DEG) hlist[atomicAdd(&nh, 1)] = i;          // (nodes are independent: any order)
        unsigned mid = __ballot_sync(0xffffffffu, deg > ATT_LANE_DEG && deg <= HEAVY_DEG);
        while (mid) {
            const int l = __ffs(mid) - 1;
            mid &= mid - 1;
            const int64_t f0 = __shfl_sync(0xffffffffu, e0, l);
            const int d = __shfl_sync(0xffffffffu, (int)deg, l);
            const float px = __shfl_sync(0xffffffffu, p.x, l), py = __shfl_sync(0xffffffffu, p.y, l);
            float2 t[HEAVY_DEG / 32];
#pragma unroll
            for (int c = 0; c < HEAVY_DEG / 32; ++c) {
                const int e = c * 32 + lane;
                const float2 o = e < d ? xy[a.cadj[f0 + e]] : make_float2(px, py);
                t[c] = make_float2(px - o.x, py - o.y);
            }
            float sx = 0.f, sy = 0.f;
#pragma unroll
            for (int c = 0; c < HEAVY_DEG / 32; ++c) {
                const int m = min(32, d - c * 32);
#pragma unroll 8
                for (int j = 0; j < m; ++j) {
                    sx -= __shfl_sync(0xffffffffu, t[c].x, j);
                    sy -= __shfl_sync(0xffffffffu, t[c].y, j);
                }
            }
            if (lane == l) {
                ax = sx;
                ay = sy;
            }
        }
        if (ok && deg <= HEAVY_DEG) {
            const float km = a.kg * a.mass[q];
            a.fa[q - a.fbase] = make_float2(ax - km * p.x, ay - km * p.y);
        }
    }
    __syncthreads();
    for (int h = 0; h < nh; ++h) {
        const int q = b.t0 + hlist[h];
        const int64_t e0 = a.coff[q], e1 = a.coff[q + 1];
        const float2 p = xy[q];
        float sx = 0.f, sy = 0.f;                                   // (thread 0)
        for (int64_t c0 = e0; c0 < e1; c0 += HEAVY_CHUNK) {
            const int64_t c1 = min(e1, c0 + HEAVY_CHUNK);
            // 256 strided sums, two a thread
#pragma unroll
            for (int u = 0; u < 256 / EX_THREADS; ++u) {
                float ax = 0.f, ay = 0.f;
                for (int64_t e = c0 + u * EX_THREADS + threadIdx.x; e < c1; e += 256) {
                    const float2 o = xy[a.cadj[e]];
                    ax -= p.x - o.x;
                    ay -= p.y - o.y;
                }
                warp_sum2(ax, ay);
                if (lane == 0) hred[u * EX_WARPS + warp] = make_float2(ax, ay);
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                float cx = 0.f, cy = 0.f;
                for (int w = 0; w < 8; ++w) {
                    cx += hred[w].x;
                    cy += hred[w].y;
                }
                sx += cx;
                sy += cy;
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            const float km = a.kg * a.mass[q];
            a.fa[q - a.fbase] = make_float2(sx - km * p.x, sy - km * p.y);
        }
    }
}

// K1 (exact), with K2 and K3 of its targets: F_rep (+ attraction + gravity,
// and the tile's swing and traction).
//
// Bound by the MUFU: one reciprocal a pair, 16 pairs per clock and SM.  A
// target's sum is a chain over its sources (in stages of 1,024, each stage's
// sum entering a compensated total), so what can be spread over the chip is
// targets times stages: a block takes EX_THREADS R targets and one stage,
// and the tile's last block to finish adds the stages in order, adds the
// attraction (a block of its own in the same launch) and sums swing and
// traction.  R = 1 for few warps (each then has a scheduler to itself), R = 2
// in packed FP32x2 arithmetic for many (less issue per pair); the sums are
// the same bit for bit.  One block per 512 targets with all their sources
// took 116 us for 2,821 nodes (6 blocks on 152 SMs).
template <int R>
__global__ void __launch_bounds__(EX_THREADS) exact_kernel(ExArgs a) {
    __shared__ float4 src[EX_STAGE + P2P_AHEAD];
    __shared__ double ws[8], wt[8];
    __shared__ bool last;
    constexpr int TT = EX_THREADS * R;
    const ExBlock b = a.blk[a.first + blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float2 *__restrict__ xy = a.xy - a.qbase;
    float sx[R], sy[R];
    if (b.s0 == b.s1) {
        tile_attraction<R>(a, b);
    } else {
        float zx[R], zy[R], cx[R], cy[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = (warp * R + r) * 32 + lane;
            const float2 p = i < b.nt ? xy[b.t0 + i] : make_float2(0.f, 0.f);
            zx[r] = p.x;
            zy[r] = p.y;
            sx[r] = sy[r] = cx[r] = cy[r] = 0.f;
        }
        const bool work = warp * R * 32 < b.nt;
        for (int s0 = b.s0; s0 < b.s1; s0 += EX_STAGE) {
            const int cnt = min(b.s1 - s0, EX_STAGE);
            __syncthreads();
#pragma unroll
            for (int k = 0; k < EX_STAGE / EX_THREADS; ++k) {
                const int j = k * EX_THREADS + threadIdx.x;
                if (j < cnt) {
                    const float2 p = xy[s0 + j];
                    src[j] = make_float4(p.x, p.y, a.mass[s0 + j], 0.f);
                }
            }
            __syncthreads();
            if (!work) continue;
            float ax[R], ay[R];
            if constexpr (R == 1) {
                ax[0] = ay[0] = 0.f;
                p2p_chain(zx[0], zy[0], src, cnt,
                          [](float dx, float dy) { return fmaf(dx, dx, fmaf(dy, dy, 1e-30f)); }, ax[0], ay[0]);
            } else {
                float2 nzx[R / 2], nzy[R / 2], gx[R / 2], gy[R / 2];
#pragma unroll
                for (int k = 0; k < R / 2; ++k) {
                    nzx[k] = make_float2(-zx[2 * k], -zx[2 * k + 1]);
                    nzy[k] = make_float2(-zy[2 * k], -zy[2 * k + 1]);
                    gx[k] = gy[k] = make_float2(0.f, 0.f);
                }
#pragma unroll 4
                for (int j = 0; j < cnt; ++j) {
                    const float4 q = src[j];
#pragma unroll
                    for (int k = 0; k < R / 2; ++k) p2p_pair2(nzx[k], nzy[k], q, gx[k], gy[k]);
                }
#pragma unroll
                for (int k = 0; k < R / 2; ++k) {
                    ax[2 * k] = -gx[k].x;
                    ax[2 * k + 1] = -gx[k].y;
                    ay[2 * k] = -gy[k].x;
                    ay[2 * k + 1] = -gy[k].y;
                }
            }
            // each stage's sum enters a compensated (Kahan) running total
#pragma unroll
            for (int r = 0; r < R; ++r) {
                float y = ax[r] - cx[r];
                float s = sx[r] + y;
                cx[r] = (s - sx[r]) - y;
                sx[r] = s;
                y = ay[r] - cy[r];
                s = sy[r] + y;
                cy[r] = (s - sy[r]) - y;
                sy[r] = s;
            }
        }
    }
    const unsigned blocks = (unsigned)b.parts + (a.att ? 1u : 0u);
    if (blocks > 1) {
        float2 *part = a.part + (size_t)b.part * TT;
        if (b.s0 != b.s1) {
#pragma unroll
            for (int r = 0; r < R; ++r)
                part[b.k * TT + (warp * R + r) * 32 + lane] = make_float2(sx[r], sy[r]);
        }
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) last = atomicAdd(&a.arrive[b.tile], 1u) == blocks - 1;
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) a.arrive[b.tile] = 0u;
        float cx[R], cy[R];
#pragma unroll
        for (int r = 0; r < R; ++r) sx[r] = sy[r] = cx[r] = cy[r] = 0.f;
        for (int k = 0; k < b.parts; ++k) {
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const float2 v = __ldcg(&part[k * TT + (warp * R + r) * 32 + lane]);
                float y = v.x - cx[r];
                float s = sx[r] + y;
                cx[r] = (s - sx[r]) - y;
                sx[r] = s;
                y = v.y - cy[r];
                s = sy[r] + y;
                cy[r] = (s - sy[r]) - y;
                sy[r] = s;
            }
        }
    }
    const bool swing = a.sw.fprev != nullptr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = (warp * R + r) * 32 + lane;
        float sw = 0.f, tr = 0.f;
        if (i < b.nt) {
            const int64_t q = b.t0 + i;
            const float m = a.mass[q], km = a.kr * m;
            const float2 t = a.att ? __ldcg(&a.fa[q - a.fbase]) : make_float2(0.f, 0.f);
            const float2 F = make_float2(fmaf(km, sx[r], t.x), fmaf(km, sy[r], t.y));
            a.f[q - a.fbase] = F;
            if (swing) fa2_swing_terms(F, a.sw.fprev[q - a.fbase], m, a.sw.variant, sw, tr);
        }
        if (swing) {
            warp_sum2(sw, tr);
            if (lane == 0) a.sw.group[(size_t)b.tile * (TT / 32) + warp * R + r] = make_float2(sw, tr);
        }
    }
    if (!swing) return;
    __threadfence();
    __syncthreads();
    const int tile0 = a.sw.tile_off[b.comp];
    if (threadIdx.x == 0)
        last = atomicAdd(&a.sw.counter[b.comp], 1u) == (unsigned)(a.sw.tile_off[b.comp + 1] - tile0) - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const float2 *group = a.sw.group + (size_t)tile0 * (TT / 32);
    const int ng = (b.n + 31) / 32, nt = (ng + 7) / 8;
#pragma unroll
    for (int u = 0; u < 256 / EX_THREADS; ++u) {
        double swg = 0.0, trc = 0.0;
        for (int k = u * EX_THREADS + (int)threadIdx.x; k < nt; k += 256) {
            double s = 0.0, t = 0.0;
            for (int w = 8 * k; w < min(8 * k + 8, ng); ++w) {
                const float2 v = __ldcg(&group[w]);         // written by other blocks: bypass L1
                s += (double)v.x;
                t += (double)v.y;
            }
            swg += s;
            trc += t;
        }
        warp_sum2(swg, trc);
        if (lane == 0) {
            ws[u * EX_WARPS + warp] = swg;
            wt[u * EX_WARPS + warp] = trc;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double swg = 0.0, trc = 0.0;
        for (int w = 0; w < 8; ++w) {
            swg += ws[w];
            trc += wt[w];
        }
        swing_finish(a.sw, b.comp, swg, trc);
    }
}

// K2: attraction and gravity written to fa (Section 3.2).  Blocks below
// n_light_blocks: one thread per node of degree <= HEAVY_DEG.  The others:
// one block per chunk of HEAVY_CHUNK adjacency entries of a node of higher
// degree; the chunk sums go to `part` and the last chunk of the node to
// finish adds them in chunk order (arrival count per node).
struct HeavyChunk {
    int32_t q;        // component-order position of the node
    int32_t h;        // index of the node among the heavy nodes
    int32_t first;    // index of the node's first chunk
    int32_t nchunk;   // chunks of the node
    int64_t e0, e1;   // adjacency entries of this chunk
};

__global__ void attraction_gravity_kernel(const float2 *__restrict__ xy, const float *__restrict__ mass,
                                          const int64_t *__restrict__ coff, const int32_t *__restrict__ cadj,
                                          int64_t q0, int64_t q1, int64_t qbase, float kg,
                                          const HeavyChunk *__restrict__ chunks, int64_t n_light_blocks,
                                          float2 *part, int *arrive, float2 *__restrict__ fa) {
    if (blockIdx.x < n_light_blocks) {
        int64_t q = q0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (q >= q1) return;
        int64_t e0 = coff[q], e1 = coff[q + 1];
        if (e1 - e0 > HEAVY_DEG) return;
        float2 p = xy[q - qbase];
        float ax = 0.f, ay = 0.f;
        for (int64_t e = e0; e < e1; ++e) {
            float2 o = xy[cadj[e] - qbase];
            ax -= p.x - o.x;
            ay -= p.y - o.y;
        }
        float km = kg * mass[q];
        fa[q - qbase] = make_float2(ax - km * p.x, ay - km * p.y);
        return;
    }
    __shared__ float rx[32], ry[32];
    __shared__ bool last;
    const int64_t k = (int64_t)blockIdx.x - n_light_blocks;
    const HeavyChunk ch = chunks[k];
    const float2 p = xy[ch.q - qbase];
    float ax = 0.f, ay = 0.f;
    for (int64_t e = ch.e0 + threadIdx.x; e < ch.e1; e += blockDim.x) {
        float2 o = xy[cadj[e] - qbase];
        ax -= p.x - o.x;
        ay -= p.y - o.y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ax += __shfl_xor_sync(0xffffffffu, ax, o);
        ay += __shfl_xor_sync(0xffffffffu, ay, o);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { rx[warp] = ax; ry[warp] = ay; }
    __syncthreads();
    if (threadIdx.x != 0) return;
    float sx = 0.f, sy = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { sx += rx[w]; sy += ry[w]; }
    part[k] = make_float2(sx, sy);
    __threadfence();
    last = atomicAdd(&arrive[ch.h], 1) == ch.nchunk - 1;
    if (!last) return;
    __threadfence();
    sx = 0.f;
    sy = 0.f;
    for (int j = 0; j < ch.nchunk; ++j) {
        const float2 v = __ldcg(&part[ch.first + j]);
        sx += v.x;
        sy += v.y;
    }
    arrive[ch.h] = 0;
    const float km = kg * mass[ch.q];
    fa[ch.q - qbase] = make_float2(sx - km * p.x, sy - km * p.y);
}

// A node of more than HEAVY_DEG adjacency entries: its place and entries
struct HeavyNode {
    int64_t q, e0, e1;
};
__global__ void heavy_kernel(const int64_t *__restrict__ coff, int64_t q0, int64_t n, HeavyNode *out, int64_t cap,
                             unsigned long long *count) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t e0 = coff[q0 + i], e1 = coff[q0 + i + 1];
    if (e1 - e0 <= HEAVY_DEG) return;
    const unsigned long long k = atomicAdd(count, 1ull);
    if ((int64_t)k < cap) out[k] = HeavyNode{q0 + i, e0, e1};
}

// K3 for the FMM's components (the exact kernel sums its own): tiles of 256
// consecutive nodes of a component, one node per thread.
__global__ void swing_traction_kernel(SwingArgs a, const Tile *__restrict__ tiles, const float2 *__restrict__ f,
                                      const float *__restrict__ mass, int64_t fbase) {
    __shared__ double ws[8], wt[8];
    __shared__ bool last;
    const Tile t = tiles[blockIdx.x];
    float sw = 0.f, tr = 0.f;
    const int i = threadIdx.x;
    if (i < (int)(t.t1 - t.t0)) {
        const int64_t q = t.t0 + i;
        fa2_swing_terms(f[q - fbase], a.fprev[q - fbase], mass[q], a.variant, sw, tr);
    }
    warp_sum2(sw, tr);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { ws[warp] = (double)sw; wt[warp] = (double)tr; }
    __syncthreads();
    const int c = t.comp, k0 = a.tile_off[c], nk = a.tile_off[c + 1] - k0;
    if (threadIdx.x == 0) {
        double s = 0.0, u = 0.0;
        for (int w = 0; w < 8; ++w) { s += ws[w]; u += wt[w]; }
        a.partial[blockIdx.x] = make_double2(s, u);
        __threadfence();
        last = atomicAdd(&a.counter[c], 1u) == (unsigned)nk - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double swg = 0.0, trc = 0.0;
    for (int k = threadIdx.x; k < nk; k += 256) {
        const double2 v = __ldcg(&a.partial[k0 + k]);   // written by other blocks: bypass L1
        swg += v.x;
        trc += v.y;
    }
    warp_sum2(swg, trc);
    __syncthreads();
    if (lane == 0) {
        ws[warp] = swg;
        wt[warp] = trc;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        swg = 0.0;
        trc = 0.0;
        for (int w = 0; w < 8; ++w) {
            swg += ws[w];
            trc += wt[w];
        }
        swing_finish(a, c, swg, trc);
    }
}

// K4: node speeds and the position update; the first thread also steps the
// loop (LOOP; a kernel without it can be profiled)
template <bool LOOP>
__global__ void update_kernel(const float2 *__restrict__ f, float2 *__restrict__ fprev, float2 *__restrict__ xy,
                              const int32_t *__restrict__ node_comp, const double *__restrict__ sg, int64_t q0,
                              int64_t q1, int64_t qbase, int64_t c0, float ks, float ksmax, int *bad,
                              LoopCtl loop) {
    if constexpr (LOOP) {
        if (blockIdx.x == 0 && threadIdx.x == 0) loop_step(loop);
    }
    int64_t q = q0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= q1) return;
    const float2 F = f[q - qbase], P = fprev[q - qbase];
    const float2 p = fa2_move(xy[q - qbase], F, P, (float)sg[node_comp[q] - c0], ks, ksmax);
    if (!isfinite(p.x) || !isfinite(p.y)) *bad = 1;
    xy[q - qbase] = p;
    fprev[q - qbase] = F;
}

inline unsigned nblocks(int64_t n, int t) { return (unsigned)std::max<int64_t>(1, (n + t - 1) / t); }

}  // namespace

// Blocks of the exact sum over the given components (indices >= c0): for each
// tile of EX_THREADS R targets one for its attraction, and one for each stage
// of its sources, or for all of them in a component of more nodes than
// split_max (the partial sums would take n^2 / 128 bytes, and there are tiles
// enough).  The order of the sums is the same either way.
struct ExactSum {
    DevBuf<ExBlock> blk;
    DevBuf<float2> part, group;
    DevBuf<unsigned> arrive;
    std::vector<int32_t> tile_off;    // per component of [c0, c1): its first tile
    int R = 1, n_blk = 0, n_tiles = 0;     // blocks of the sum (the tiles' attraction blocks come before them)

    // reps: every tile so many times (each copy writes the same forces)
    void make(bgl_graph *g, int64_t c0, int64_t c1, const std::vector<int64_t> &comps, int reps = 1) {
        int64_t split_max = EX_SPLIT_FREE_N, bytes = 0;
        for (auto it = comps.rbegin(); it != comps.rend(); ++it) {            // (sizes descend)
            const int64_t n = g->h_comp_off[*it + 1] - g->h_comp_off[*it];
            if (n <= EX_SPLIT_FREE_N) continue;
            bytes += (n + 255) / 256 * 256 * ((n + EX_STAGE - 1) / EX_STAGE) * (int64_t)sizeof(float2) * reps;
            if (n > EX_SPLIT_MAX_N || bytes > EX_PART_BYTES) {
                split_max = std::min(split_max, n - 1);                       // (none of this size)
                break;
            }
            split_max = n;
        }
        auto parts_of = [split_max](int64_t n) {
            return n <= split_max ? (n + EX_STAGE - 1) / EX_STAGE : int64_t(1);
        };
        int64_t wide = 0;
        for (int64_t c : comps) {
            const int64_t n = g->h_comp_off[c + 1] - g->h_comp_off[c];
            wide += (n + 63) / 64 * parts_of(n) * reps;
        }
        R = wide >= BGL_EXACT_WIDE_WARPS ? 2 : 1;
        const int64_t tt = EX_THREADS * R;
        std::vector<ExBlock> att, sum;
        tile_off.assign(c1 - c0 + 1, 0);
        int32_t tile = 0, units = 0;
        size_t next = 0;
        for (int64_t c = c0; c < c1; ++c) {
            tile_off[c - c0] = tile;
            if (next >= comps.size() || comps[next] != c) continue;
            ++next;
            const int64_t a = g->h_comp_off[c], n = g->h_comp_off[c + 1] - a, parts = parts_of(n);
            for (int r = 0; r < reps; ++r)
                for (int64_t t = 0; t < n; t += tt, ++tile, units += (int32_t)parts) {
                    ExBlock b;
                    b.t0 = (int32_t)(a + t);
                    b.nt = (int32_t)std::min(tt, n - t);
                    b.s0 = b.s1 = 0;
                    b.comp = (int32_t)(c - c0);
                    b.tile = tile;
                    b.k = -1;
                    b.parts = (int32_t)parts;
                    b.part = units;
                    b.n = (int32_t)n;
                    att.push_back(b);
                    for (int64_t k = 0; k < parts; ++k) {
                        b.k = (int32_t)k;
                        b.s0 = (int32_t)(a + k * EX_STAGE);
                        b.s1 = (int32_t)(a + (k + 1 < parts ? (k + 1) * EX_STAGE : n));
                        sum.push_back(b);
                    }
                }
        }
        tile_off[c1 - c0] = tile;
        n_blk = (int)sum.size();
        n_tiles = tile;
        if (!n_blk) return;
        att.insert(att.end(), sum.begin(), sum.end());
        Allocator *A = g->ctx->alloc;
        cudaStream_t s = g->ctx->stream;
        blk.reset(A, att.size());
        part.reset(A, (size_t)units * tt);
        group.reset(A, (size_t)tile * (tt / 32));
        arrive.reset(A, tile);
        BGL_CUDA(cudaMemcpyAsync(blk.p, att.data(), sizeof(ExBlock) * att.size(), cudaMemcpyHostToDevice, s));
        BGL_CUDA(cudaMemsetAsync(arrive.p, 0, sizeof(unsigned) * tile, s));
        BGL_CUDA(cudaStreamSynchronize(s));      // att goes out of scope
    }

    // F_rep, or with fa (scratch) the total force; swing and traction where sw.fprev is set
    void launch(const bgl_graph *g, const bgl_params *p, const float2 *xy, int64_t qbase, float2 *f, int64_t fbase,
                float2 *fa, const SwingArgs &sw, cudaStream_t s) const {
        if (!n_blk) return;
        ExArgs a;
        a.blk = blk.p;
        a.att = fa != nullptr;
        a.first = a.att ? 0 : n_tiles;
        a.xy = xy;
        a.mass = g->mass.p;
        a.coff = g->coff.p;
        a.cadj = g->cadj.p;
        a.qbase = qbase;
        a.fbase = fbase;
        a.kr = (float)p->kr;
        a.kg = (float)p->kg;
        a.part = part.p;
        a.arrive = arrive.p;
        a.fa = fa;
        a.f = f;
        a.sw = sw;
        a.sw.group = group.p;
        const unsigned blocks = (unsigned)(n_blk + (a.att ? n_tiles : 0));
        if (R == 1) exact_kernel<1><<<blocks, EX_THREADS, 0, s>>>(a);
        else exact_kernel<2><<<blocks, EX_THREADS, 0, s>>>(a);
        BGL_LAUNCH_CHECK();
    }
};

bool use_fmm(const bgl_params *p, int64_t n) {
    if (p->repulsion == BGL_REP_FMM) return true;
    if (p->repulsion == BGL_REP_EXACT) return false;
    return n >= p->fmm_min_nodes;
}

// Measured exact/FMM crossover (repulsion AUTO with fmm_min_nodes = -1).
// Components below TUNE_LO nodes take the exact sum, those of TUNE_HI or
// more the FMM.  In between, the first component of each size octave that a
// context meets is measured at its initial positions: one FMM evaluation
// (its cost as it runs, one component after another on the stream), and
// the exact sum's pair rate with the component's tiles repeated until they
// fill every SM (the rate the exact tiles of a batch of components reach
// together); the FMM is kept for that octave (and that p and leaf size) if
// its evaluation takes less than n^2 pairs at that rate.
constexpr int64_t TUNE_LO = 2048, TUNE_HI = 1 << 17;

static bool use_fmm_for(bgl_graph *g, const bgl_params *p, int64_t c) {
    const int64_t n = g->h_comp_off[c + 1] - g->h_comp_off[c];
    if (p->repulsion != BGL_REP_AUTO || p->fmm_min_nodes >= 0) return use_fmm(p, n);
    if (n < TUNE_LO) return false;
    if (n >= TUNE_HI) return true;
    bgl_ctx *ctx = g->ctx;
    const int key = (int)std::log2((double)n) * 10000 + p->fmm_p * 300 + p->leaf_size;
    {
        std::lock_guard<std::mutex> lk(ctx->tune_mu);
        auto it = ctx->tune_fmm.find(key);
        if (it != ctx->tune_fmm.end()) return it->second;
    }
    cudaStream_t s = ctx->stream;
    const int64_t q0 = g->h_comp_off[c], q1 = g->h_comp_off[c + 1];
    DevBuf<float2> xy(ctx->alloc, n), f(ctx->alloc, n);
    init_positions(g, p, xy.p, q0, q1);
    // repeated until there are eight blocks per SM (each copy writes the same forces)
    ExactSum ex;
    ex.make(g, c, c + 1, {c});
    const int reps = std::max<int>(1, (8 * ctx->num_sms + ex.n_blk - 1) / ex.n_blk);
    ex.make(g, c, c + 1, {c}, reps);
    FmmPlan *pl = fmm_create(g, p, c);
    cudaEvent_t e[4] = {nullptr, nullptr, nullptr, nullptr};
    float ms_fmm = 0.f, ms_exact = 0.f;
    try {
        for (auto &ev : e) BGL_CUDA(cudaEventCreate(&ev));
        fmm_repulsion(pl, xy.p, q0, f.p, q0);
        BGL_CUDA(cudaEventRecord(e[0], s));
        fmm_repulsion(pl, xy.p, q0, f.p, q0);
        BGL_CUDA(cudaEventRecord(e[1], s));
        ex.launch(g, p, xy.p, q0, f.p, q0, nullptr, SwingArgs{}, s);
        BGL_CUDA(cudaEventRecord(e[2], s));
        ex.launch(g, p, xy.p, q0, f.p, q0, nullptr, SwingArgs{}, s);
        BGL_CUDA(cudaEventRecord(e[3], s));
        BGL_CUDA(cudaEventSynchronize(e[3]));
        BGL_CUDA(cudaEventElapsedTime(&ms_fmm, e[0], e[1]));
        BGL_CUDA(cudaEventElapsedTime(&ms_exact, e[2], e[3]));
        const int err = fmm_error(pl);
        if (err & 1) fail(BGL_ETIMEOUT, "fmm: a bounded device-side wait gave up");
        if (err & 8) fail(BGL_ENUMERIC, "fmm: non-finite positions");
        if (err) fail(BGL_ENOMEM, "fmm: tree or list capacity exceeded (error bits " + std::to_string(err) + ")");
    } catch (...) {
        for (auto ev : e)
            if (ev) cudaEventDestroy(ev);
        fmm_destroy(pl);
        throw;
    }
    for (auto ev : e) cudaEventDestroy(ev);
    fmm_destroy(pl);
    // the exact sum of this component alone, at the batched pair rate
    const double exact_ms = (double)ms_exact / reps;
    const bool fmm = ms_fmm < exact_ms;
    std::lock_guard<std::mutex> lk(ctx->tune_mu);
    ctx->tune_fmm[key] = fmm;
    return fmm;
}

// Everything one set of ForceAtlas2 components needs across iterations.
struct Fa2Run {
    bgl_graph *g;
    const bgl_params *p;
    float2 *xy;
    int64_t qbase, c0, c1, q0, q1;
    ExactSum exact;
    DevBuf<Tile> red_tiles;       // swing/traction tiles of the FMM's components
    DevBuf<int32_t> red_tile_off, ex_tile_off;
    int n_red_tiles = 0;
    int64_t q_fmm = 0;            // end of the last FMM component (the attraction kernel's range is [q0, q_fmm))
    DevBuf<float2> f, fprev, fa;
    DevBuf<double2> partial;
    DevBuf<double> sg;
    DevBuf<unsigned> counter;
    DevBuf<int> iter;
    DevBuf<int> loop;              // iterations done by the device-side loop of one graph launch
    DevBuf<HeavyChunk> chunks;
    DevBuf<float2> chunk_part;
    DevBuf<int> chunk_arrive;
    int64_t n_chunks = 0;
    std::vector<FmmPlan *> fmm;   // one per FMM component
    std::vector<int64_t> fmm_comp;
    PoolStream side;              // attraction + gravity, beside the repulsion
    PoolEvent ev_fork, ev_fa;
    // A run whose only component is on the FMM path iterates fused: the FMM's
    // combine pass sums swing and traction and sets s_G, and one kernel moves
    // the points and makes the next evaluation's root square (no swing/traction
    // kernel, no bounding-box kernel).  BGL_FUSED_ITERATION=0 turns it off.
    bool fused = false;

    void enable_fuse(double *d_stats) {
        if (!fused) {
            const char *v = std::getenv("BGL_FUSED_ITERATION");
            if (v && v[0] == '0') return;
            if (fmm.size() != 1 || exact.n_blk != 0 || c1 - c0 != 1) return;
        }
        FmmFuse fz;
        fz.fprev = fprev.p;
        fz.variant = p->swing_variant;
        fz.tau = p->tau;
        fz.sg = sg.p;
        fz.stats = d_stats;
        fz.iter = iter.p;
        fz.ks = (float)p->ks;
        fz.ksmax = (float)p->ksmax;
        fz.bad = g->ctx->d_flag + 1;
        fmm_fuse(fmm[0], fz);
        fused = true;
    }

    Fa2Run(bgl_graph *g_, const bgl_params *p_, float2 *xy_, int64_t qbase_, int64_t c0_, int64_t c1_)
        : g(g_), p(p_), xy(xy_), qbase(qbase_), c0(c0_), c1(c1_) {
        Allocator *A = g->ctx->alloc;
        cudaStream_t s = g->ctx->stream;
        q0 = g->h_comp_off[c0];
        q1 = g->h_comp_off[c1];
        const int64_t n = q1 - q0;
        std::vector<Tile> red;
        std::vector<int64_t> ex_comps;
        std::vector<int32_t> roff(1, 0);
        q_fmm = q0;
        for (int64_t c = c0; c < c1; ++c) {
            int64_t a = g->h_comp_off[c], b = g->h_comp_off[c + 1];
            if (use_fmm_for(g, p, c)) {
                fmm.push_back(fmm_create(g, p, c));
                fmm_comp.push_back(c);
                q_fmm = b;
                for (int64_t t = a; t < b; t += RED_TILE)
                    red.push_back(Tile{(int32_t)(c - c0), 0, t, std::min(b, t + RED_TILE)});
            } else {
                ex_comps.push_back(c);
            }
            roff.push_back((int32_t)red.size());
        }
        if (!ex_comps.empty()) {
            exact.make(g, c0, c1, ex_comps);
            ex_tile_off.reset(A, exact.tile_off.size());
            BGL_CUDA(cudaMemcpyAsync(ex_tile_off.p, exact.tile_off.data(), sizeof(int32_t) * exact.tile_off.size(),
                                     cudaMemcpyHostToDevice, s));
        }
        n_red_tiles = (int)red.size();
        if (n_red_tiles > 0) {
            red_tiles.reset(A, red.size());
            red_tile_off.reset(A, roff.size());
            BGL_CUDA(cudaMemcpyAsync(red_tiles.p, red.data(), sizeof(Tile) * red.size(), cudaMemcpyHostToDevice, s));
            BGL_CUDA(cudaMemcpyAsync(red_tile_off.p, roff.data(), sizeof(int32_t) * roff.size(),
                                     cudaMemcpyHostToDevice, s));
            partial.reset(A, red.size());
        }
        fa.reset(A, n);
        f.reset(A, n);
        fprev.reset(A, n);
        BGL_CUDA(cudaMemsetAsync(fprev.p, 0, sizeof(float2) * n, s));
        std::vector<double> ones(c1 - c0, 1.0);
        sg.reset(A, c1 - c0);
        BGL_CUDA(cudaMemcpyAsync(sg.p, ones.data(), sizeof(double) * ones.size(), cudaMemcpyHostToDevice, s));
        counter.reset(A, std::max<int64_t>(c1 - c0, 1));
        BGL_CUDA(cudaMemsetAsync(counter.p, 0, sizeof(unsigned) * std::max<int64_t>(c1 - c0, 1), s));
        iter.reset(A, 1);
        BGL_CUDA(cudaMemsetAsync(iter.p, 0, sizeof(int), s));
        loop.reset(A, 1);
        if (!fmm.empty()) heavy_setup();
        side.take(g->ctx);
        ev_fork.take(g->ctx);
        ev_fa.take(g->ctx);
        BGL_CUDA(cudaStreamSynchronize(s));
    }
    ~Fa2Run() {
        for (auto *pl : fmm) fmm_destroy(pl);
    }

    // the FMM components' nodes of high degree: chunks of HEAVY_CHUNK adjacency entries
    void heavy_setup() {
        Allocator *A = g->ctx->alloc;
        cudaStream_t s = g->ctx->stream;
        const int64_t nf = q_fmm - q0;
        // the count and the first of them in one copy; there are at most 2 E / HEAVY_DEG
        constexpr int64_t FIRST = 256;
        const int64_t cap = std::max<int64_t>(FIRST, 2 * g->n_undir / HEAVY_DEG + 1);
        DevBuf<HeavyNode> heavy(A, cap + 1);
        unsigned long long *count = reinterpret_cast<unsigned long long *>(heavy.p);
        BGL_CUDA(cudaMemsetAsync(count, 0, sizeof(unsigned long long), s));
        heavy_kernel<<<nblocks(nf, 256), 256, 0, s>>>(g->coff.p, q0, nf, heavy.p + 1, cap, count);
        BGL_LAUNCH_CHECK();
        std::vector<HeavyNode> hn(FIRST + 1);
        BGL_CUDA(cudaMemcpyAsync(hn.data(), heavy.p, sizeof(HeavyNode) * hn.size(), cudaMemcpyDeviceToHost, s));
        BGL_CUDA(cudaStreamSynchronize(s));
        const int32_t nh = (int32_t) * reinterpret_cast<unsigned long long *>(hn.data());
        if (nh > FIRST) {
            hn.resize(nh + 1);
            BGL_CUDA(cudaMemcpyAsync(hn.data(), heavy.p, sizeof(HeavyNode) * hn.size(), cudaMemcpyDeviceToHost, s));
            BGL_CUDA(cudaStreamSynchronize(s));
        }
        hn.erase(hn.begin());
        hn.resize(nh);
        std::sort(hn.begin(), hn.end(), [](const HeavyNode &x, const HeavyNode &y) { return x.q < y.q; });
        std::vector<HeavyChunk> hc;
        for (int32_t h = 0; h < nh; ++h) {
            const int32_t first = (int32_t)hc.size();
            const int32_t nchunk = (int32_t)((hn[h].e1 - hn[h].e0 + HEAVY_CHUNK - 1) / HEAVY_CHUNK);
            for (int32_t j = 0; j < nchunk; ++j)
                hc.push_back(HeavyChunk{(int32_t)hn[h].q, h, first, nchunk, hn[h].e0 + (int64_t)j * HEAVY_CHUNK,
                                        std::min<int64_t>(hn[h].e1, hn[h].e0 + (int64_t)(j + 1) * HEAVY_CHUNK)});
        }
        n_chunks = (int64_t)hc.size();
        chunks.reset(A, hc.size());
        chunk_part.reset(A, hc.size());
        chunk_arrive.reset(A, std::max<int32_t>(nh, 1));
        BGL_CUDA(cudaMemsetAsync(chunk_arrive.p, 0, sizeof(int) * std::max<int32_t>(nh, 1), s));
        if (!hc.empty())
            BGL_CUDA(cudaMemcpyAsync(chunks.p, hc.data(), sizeof(HeavyChunk) * hc.size(), cudaMemcpyHostToDevice, s));
    }

    // device-side failures of the FMM (bounded waits, capacities)
    void check_fmm() {
        for (auto *pl : fmm) {
            int e = fmm_error(pl);
            if (e & 1) fail(BGL_ETIMEOUT, "fmm: a bounded device-side wait gave up");
            if (e & 8) fail(BGL_ENUMERIC, "fmm: non-finite positions");
            if (e) fail(BGL_ENOMEM, "fmm: tree or list capacity exceeded (error bits " + std::to_string(e) + ")");
        }
    }

    SwingArgs swing_args(double *d_stats) const {
        SwingArgs a;
        a.fprev = fprev.p;
        a.variant = p->swing_variant;
        a.tau = p->tau;
        a.partial = partial.p;
        a.group = nullptr;
        a.tile_off = red_tile_off.p;
        a.sg = sg.p;
        a.counter = counter.p;
        a.stats = d_stats;
        a.iter = iter.p;
        return a;
    }

    // K1 + K2: f <- F (what 0) or F_rep (what 1).  The FMM's K2 runs on the
    // side stream from the start; its kernels that write f last wait for it
    // (event ev_fa) and add fa.  The exact kernel adds its targets' K2 and,
    // with `sw`, sums their K3.
    void forces(int what, const SwingArgs *sw = nullptr) {
        cudaStream_t s = g->ctx->stream;
        const bool att = what == 0;
        if (att && !fmm.empty()) {
            BGL_RANGE("ForceAtlas2: attraction and gravity (Section 3.2)");
            BGL_CUDA(cudaEventRecord(ev_fork, s));
            BGL_CUDA(cudaStreamWaitEvent(side, ev_fork, 0));
            int64_t nl = nblocks(q_fmm - q0, 256);
            attraction_gravity_kernel<<<(unsigned)(nl + n_chunks), 256, 0, side>>>(
                xy, g->mass.p, g->coff.p, g->cadj.p, q0, q_fmm, qbase, (float)p->kg, chunks.p, nl, chunk_part.p,
                chunk_arrive.p, fa.p - (q0 - qbase));
            BGL_LAUNCH_CHECK();
            BGL_CUDA(cudaEventRecord(ev_fa, side));
        }
        for (size_t k = 0; k < fmm.size(); ++k) {
            BGL_RANGE("ForceAtlas2: repulsion by the FMM (Section 3.2.1)");
            fmm_repulsion(fmm[k], xy, qbase, f.p, q0, att ? fa.p : nullptr, att ? (cudaEvent_t)ev_fa : nullptr);
        }
        if (att && !fmm.empty()) BGL_CUDA(cudaStreamWaitEvent(s, ev_fa, 0));
        if (exact.n_blk > 0) {
            BGL_RANGE("ForceAtlas2: exact repulsion (Section 3.2)");
            SwingArgs a{};
            if (sw) {
                a = *sw;
                a.tile_off = ex_tile_off.p;
            }
            exact.launch(g, p, xy, qbase, f.p, q0, att ? fa.p : nullptr, a, s);
        }
    }

    // one full iteration (K1..K4); loop: the device-side loop's control, done by K4
    void iteration(double *d_stats, const LoopCtl &loop_ctl = LoopCtl{}) {
        BGL_RANGE("ForceAtlas2 iteration: forces, swing/traction, update (Section 3.2)");
        cudaStream_t s = g->ctx->stream;
        if (fused) {
            // K3 in the FMM's combine pass, K4 with the next root square
            forces(0);
            BGL_RANGE("ForceAtlas2: node update (Section 3.2)");
            fmm_update_root(fmm[0], xy, qbase, f.p, fprev.p, q0, loop_ctl);
            return;
        }
        const SwingArgs a = swing_args(d_stats);
        forces(0, &a);
        {
            BGL_RANGE("ForceAtlas2: swing and traction (Section 3.2)");
            if (n_red_tiles > 0) {
                swing_traction_kernel<<<n_red_tiles, 256, 0, s>>>(a, red_tiles.p, f.p, g->mass.p, q0);
                BGL_LAUNCH_CHECK();
            }
        }
        BGL_RANGE("ForceAtlas2: node update (Section 3.2)");
        (loop_ctl.count ? update_kernel<true> : update_kernel<false>)<<<nblocks(q1 - q0, 256), 256, 0, s>>>(
            f.p - (q0 - qbase), fprev.p - (q0 - qbase), xy, g->node_comp.p, sg.p, q0, q1, qbase, c0, (float)p->ks,
            (float)p->ksmax, g->ctx->d_flag + 1, loop_ctl);
        BGL_LAUNCH_CHECK();
    }
};

// With BGL_HOST_LOOP=1 in the environment, the iterations are launched
// from the host as one captured-iteration graph each instead of a device-side
// loop: profilers that cannot look inside graphs with conditional nodes can
// then see every kernel.  The results are the same.
static bool host_loop() {
    const char *v = std::getenv("BGL_HOST_LOOP");
    return v && v[0] == '1';
}

static void run_iterations_host(Fa2Run &run, int iters, double *d_stats, const SideWork &side) {
    bgl_ctx *ctx = run.g->ctx;
    cudaStream_t s = ctx->stream;
    cudaEvent_t side_done = nullptr;
    if (side) {
        // the side work on its own stream beside the iterations, joined after them
        BGL_CUDA(cudaEventCreateWithFlags(&side_done, cudaEventDisableTiming));
        BGL_CUDA(cudaEventRecord(run.ev_fork, s));
        BGL_CUDA(cudaStreamWaitEvent(run.side, run.ev_fork, 0));
        try {
            side.enqueue(run.side);
            BGL_CUDA(cudaEventRecord(side_done, run.side));
        } catch (...) {
            cudaEventDestroy(side_done);
            throw;
        }
    }
    struct EventGuard {
        cudaEvent_t e;
        ~EventGuard() { if (e) cudaEventDestroy(e); }
    } side_guard{side_done};
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    const int64_t before = launch_count();
    BGL_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    ctx->alloc->forbid = true;
    try {
        run.iteration(d_stats);
    } catch (...) {
        ctx->alloc->forbid = false;
        cudaGraph_t tmp = nullptr;
        cudaStreamEndCapture(s, &tmp);
        if (tmp) cudaGraphDestroy(tmp);
        throw;
    }
    ctx->alloc->forbid = false;
    BGL_CUDA(cudaStreamEndCapture(s, &graph));
    const int64_t per_iter = launch_count() - before;
    count_launches(-per_iter);
    try {
        BGL_CUDA(cudaGraphInstantiate(&exec, graph, 0));
    } catch (...) {
        cudaGraphDestroy(graph);
        throw;
    }
    cudaGraphDestroy(graph);
    try {
        // a fused iteration finds the root square made by the previous one;
        // the first one's comes from the current positions
        if (run.fused) fmm_root(run.fmm[0], run.xy, run.qbase);
        for (int k = 0; k < iters; ++k) BGL_CUDA(cudaGraphLaunch(exec, s));
    } catch (...) {
        cudaGraphExecDestroy(exec);
        throw;
    }
    count_launches(per_iter * iters);
    if (side_done) BGL_CUDA(cudaStreamWaitEvent(s, side_done, 0));
    BGL_CUDA(cudaMemcpyAsync(ctx->h_flag + 1, ctx->d_flag + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    BGL_CUDA(cudaStreamSynchronize(s));
    cudaGraphExecDestroy(exec);
    run.check_fmm();
    if (ctx->h_flag[1]) fail(BGL_ENUMERIC, "fa2: a position became non-finite");
}

// Iterations per turn of the device-side loop.  A turn costs some 4 us beside
// its kernels: of a 25 us iteration of exact sums four to a turn save 3.5 us
// (871 nodes: 24.8 us an iteration with one, 22.6 two, 21.5 four, 20.9 eight).
// Every captured iteration also costs the instantiation of its kernels, some
// 30 us for an FMM iteration, which two to a turn win back in 24 iterations.
static int loop_unroll(const Fa2Run &run, int iters) { return run.fmm.empty() ? 4 : (iters >= 24 ? 2 : 1); }

// Gives every kernel of a graph the shared-memory split that the Kamada-Kawai
// kernels ask for.  An SM changes its split only when it is empty: beside
// Kamada-Kawai classes an exact sum that wants another one keeps SMs from
// them, and their blocks pile up on the others (50 exact iterations of 6,000
// nodes beside 1,000 components of 3 to 200 nodes: 27.8 to 68 ms without this,
// 27 to 31 with it; beside 20,000 64 to 89 and 35 to 45).  The FMM's kernels
// are better with their own (10,000 nodes alone: 4.2 ms, 4.5 with this one;
// 100,000 beside 100,000 components of 3 to 30: 13.65 and 13.96).
static void widest_shared_memory(cudaGraph_t graph) {
    size_t n = 0;
    BGL_CUDA(cudaGraphGetNodes(graph, nullptr, &n));
    std::vector<cudaGraphNode_t> nodes(n);
    if (n) BGL_CUDA(cudaGraphGetNodes(graph, nodes.data(), &n));
    cudaLaunchAttributeValue v = {};
    v.sharedMemCarveout = (unsigned)cudaSharedmemCarveoutMaxShared;
    for (cudaGraphNode_t nd : nodes) {
        cudaGraphNodeType t;
        BGL_CUDA(cudaGraphNodeGetType(nd, &t));
        if (t == cudaGraphNodeTypeKernel)
            BGL_CUDA(cudaGraphKernelNodeSetAttribute(nd, cudaLaunchAttributePreferredSharedMemoryCarveout, &v));
    }
}

// `n` iterations captured on s into graph `into` (null: a new graph, which
// is returned); loop: stepped by the last one.  Adds the kernels to `kernels`.
static cudaGraph_t capture_iterations(Fa2Run &run, double *d_stats, int n, cudaGraph_t into, const LoopCtl &loop,
                                      int64_t &kernels) {
    bgl_ctx *ctx = run.g->ctx;
    cudaStream_t s = ctx->stream;
    const int64_t before = launch_count();
    if (into) {
        BGL_CUDA(cudaStreamBeginCaptureToGraph(s, into, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
    } else {
        BGL_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    }
    ctx->alloc->forbid = true;
    cudaGraph_t captured = nullptr;
    try {
        for (int k = 0; k < n; ++k) run.iteration(d_stats, k + 1 < n ? LoopCtl{} : loop);
    } catch (...) {
        ctx->alloc->forbid = false;
        cudaStreamEndCapture(s, &captured);
        if (captured && !into) cudaGraphDestroy(captured);
        throw;
    }
    ctx->alloc->forbid = false;
    BGL_CUDA(cudaStreamEndCapture(s, &captured));
    // captured launches run only when the graph does
    kernels = launch_count() - before;
    count_launches(-kernels);
    return captured;
}

// All `iters` iterations of `run` in one graph launch: the graph holds a
// WHILE conditional node whose body is some captured iterations, the last
// kernel of which counts them and clears the condition after the last, so
// the loop runs on the device without the host; the iterations that are left
// over come before it.  Nothing may allocate while a capture is open.
static void run_iterations(Fa2Run &run, int iters, double *d_stats, const SideWork &side = SideWork()) {
    bgl_ctx *ctx = run.g->ctx;
    cudaStream_t s = ctx->stream;
    if (iters <= 0) {
        if (side) side.enqueue(s);
        return;
    }
    BGL_CUDA(cudaMemsetAsync(ctx->d_flag + 1, 0, sizeof(int), s));
    BGL_CUDA(cudaMemsetAsync(run.iter.p, 0, sizeof(int), s));
    BGL_CUDA(cudaMemsetAsync(run.loop.p, 0, sizeof(int), s));
    run.enable_fuse(d_stats);
    if (host_loop()) {
        run_iterations_host(run, iters, d_stats, side);
        return;
    }
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    BGL_CUDA(cudaGraphCreate(&graph, 0));
    int64_t kernels = 0;
    const bool widest = run.exact.n_blk > 0 && side;
    try {
        const int unroll = loop_unroll(run, iters), turns = iters / unroll, rest = iters - turns * unroll;
        cudaGraphNode_t rnode = nullptr;
        if (rest > 0) {
            struct Child {
                cudaGraph_t g;
                ~Child() { cudaGraphDestroy(g); }
            } child{capture_iterations(run, d_stats, rest, nullptr, LoopCtl{}, kernels)};
            if (widest) widest_shared_memory(child.g);
            BGL_CUDA(cudaGraphAddChildGraphNode(&rnode, graph, nullptr, 0, child.g));
        }
        if (turns > 0) {
            LoopCtl ctl;
            BGL_CUDA(cudaGraphConditionalHandleCreate(&ctl.h, graph, 1, cudaGraphCondAssignDefault));
            ctl.count = run.loop.p;
            ctl.iters = turns;
            cudaGraphNodeParams cp = {};
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = ctl.h;
            cp.conditional.type = cudaGraphCondTypeWhile;
            cp.conditional.size = 1;
            cudaGraphNode_t cnode;
            BGL_CUDA(cudaGraphAddNode(&cnode, graph, rnode ? &rnode : nullptr, nullptr, rnode ? 1 : 0, &cp));
            int64_t per_turn = 0;
            capture_iterations(run, d_stats, unroll, cp.conditional.phGraph_out[0], ctl, per_turn);
            kernels += per_turn * turns;
            if (widest) widest_shared_memory(cp.conditional.phGraph_out[0]);
        }
        if (side) {
            // the side work, captured on the run's side stream (it may fork
            // to streams of its own), becomes a child graph beside the loop
            cudaGraph_t child = nullptr;
            BGL_CUDA(cudaStreamBeginCapture(run.side, cudaStreamCaptureModeThreadLocal));
            ctx->alloc->forbid = true;
            try {
                side.enqueue(run.side);
            } catch (...) {
                ctx->alloc->forbid = false;
                cudaGraph_t tmp = nullptr;
                cudaStreamEndCapture(run.side, &tmp);
                if (tmp) cudaGraphDestroy(tmp);
                throw;
            }
            ctx->alloc->forbid = false;
            BGL_CUDA(cudaStreamEndCapture(run.side, &child));
            cudaGraphNode_t cn;
            const cudaError_t e = cudaGraphAddChildGraphNode(&cn, graph, nullptr, 0, child);
            cudaGraphDestroy(child);
            BGL_CUDA(e);
        }
        BGL_CUDA(cudaGraphInstantiate(&exec, graph, 0));
    } catch (...) {
        cudaGraphDestroy(graph);
        throw;
    }
    cudaGraphDestroy(graph);
    count_launches(kernels);
    try {
        if (run.fused) fmm_root(run.fmm[0], run.xy, run.qbase);
        BGL_CUDA(cudaGraphLaunch(exec, s));
    } catch (...) {
        cudaGraphExecDestroy(exec);
        throw;
    }
    BGL_CUDA(cudaMemcpyAsync(ctx->h_flag + 1, ctx->d_flag + 1, sizeof(int), cudaMemcpyDeviceToHost, s));
    BGL_CUDA(cudaStreamSynchronize(s));
    cudaGraphExecDestroy(exec);
    run.check_fmm();
    if (ctx->h_flag[1]) fail(BGL_ENUMERIC, "fa2: a position became non-finite");
}

void fa2_layout(bgl_graph *g, const bgl_params *p, float2 *xy, int64_t qbase, int64_t c0, int64_t c1, int iters,
                double *d_stats, const SideWork &side) {
    if (c1 <= c0 || iters <= 0) {
        if (side) side.enqueue(g->ctx->stream);
        return;
    }
    BGL_RANGE("ForceAtlas2 iterations (Section 3.2)");
    Fa2Run run(g, p, xy, qbase, c0, c1);
    for (FmmPlan *pl : run.fmm) fmm_crowded(pl, side.fills(g->ctx));
    run_iterations(run, iters, d_stats, side);
}

// ---------------------------------------------------------------- resumable runs

namespace {

// 64-bit FNV-1a over a byte range
uint64_t fnv1a(uint64_t h, const void *data, size_t len) {
    const unsigned char *b = static_cast<const unsigned char *>(data);
    for (size_t i = 0; i < len; ++i) {
        h ^= b[i];
        h *= 0x100000001b3ull;
    }
    return h;
}

// Identity of component c of g: its size, position in the component order,
// node ids and adjacency rows (a checkpoint loads only into the same graph).
uint64_t component_fingerprint(bgl_graph *g, int64_t c) {
    const int64_t q0 = g->h_comp_off[c], q1 = g->h_comp_off[c + 1], n = q1 - q0;
    std::vector<int32_t> nodes(n);
    std::vector<int64_t> coff(n + 1);
    cudaStream_t s = g->ctx->stream;
    BGL_CUDA(cudaMemcpyAsync(nodes.data(), g->nodes.p + q0, sizeof(int32_t) * n, cudaMemcpyDeviceToHost, s));
    BGL_CUDA(cudaMemcpyAsync(coff.data(), g->coff.p + q0, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, s));
    BGL_CUDA(cudaStreamSynchronize(s));
    const int64_t e0 = coff[0], e1 = coff[n];
    std::vector<int32_t> cadj(e1 - e0);
    if (e1 > e0)
        BGL_CUDA(cudaMemcpyAsync(cadj.data(), g->cadj.p + e0, sizeof(int32_t) * (e1 - e0), cudaMemcpyDeviceToHost, s));
    BGL_CUDA(cudaStreamSynchronize(s));
    for (auto &o : coff) o -= e0;
    uint64_t h = 0xcbf29ce484222325ull;
    const int64_t head[4] = {g->n, g->n_undir, c, n};
    h = fnv1a(h, head, sizeof(head));
    h = fnv1a(h, nodes.data(), sizeof(int32_t) * n);
    h = fnv1a(h, coff.data(), sizeof(int64_t) * (n + 1));
    h = fnv1a(h, cadj.data(), sizeof(int32_t) * cadj.size());
    return h;
}

// checkpoint layout: this header, then n float2 positions and n float2 F_{t-1}
struct StateHeader {
    char magic[8];
    uint32_t version;
    uint32_t header_bytes;
    int64_t n_nodes, n_undir, comp, comp_nodes;
    uint64_t fingerprint;
    int64_t iters_done;
    double sg;
    int32_t fmm_sortskip;          // FMM sort passes the next evaluation skips (-1: exact repulsion)
    int32_t pad;
    bgl_params params;
};
constexpr char STATE_MAGIC[8] = {'B', 'G', 'L', 'F', 'A', '2', 'S', 'T'};
constexpr uint32_t STATE_VERSION = 1;

}  // namespace

struct Fa2Session {
    bgl_graph *g = nullptr;
    bgl_params p;                  // owned copy (the run keeps a pointer to it)
    int64_t c = 0, q0 = 0, n = 0;
    int64_t iters_done = 0;
    uint64_t fingerprint = 0;
    DevBuf<float2> xy;             // positions, xy[q - q0]
    Fa2Run *run = nullptr;
    ~Fa2Session() { delete run; }
};

static Fa2Session *session_new(bgl_graph *g, const bgl_params *p, int64_t c) {
    Fa2Session *s = new Fa2Session();
    try {
        s->g = g;
        s->p = *p;
        s->c = c;
        s->q0 = g->h_comp_off[c];
        s->n = g->h_comp_off[c + 1] - s->q0;
        s->xy.reset(g->ctx->alloc, std::max<int64_t>(s->n, 1));
        s->run = new Fa2Run(g, &s->p, s->xy.p, s->q0, c, c + 1);
        s->fingerprint = component_fingerprint(g, c);
    } catch (...) {
        delete s;
        throw;
    }
    return s;
}

Fa2Session *fa2_session_create(bgl_graph *g, const bgl_params *p, int64_t c, const float2 *h_xy) {
    Fa2Session *s = session_new(g, p, c);
    try {
        BGL_CUDA(cudaMemcpyAsync(s->xy.p, h_xy, sizeof(float2) * s->n, cudaMemcpyHostToDevice, g->ctx->stream));
        BGL_CUDA(cudaStreamSynchronize(g->ctx->stream));
    } catch (...) {
        delete s;
        throw;
    }
    return s;
}

void fa2_session_destroy(Fa2Session *s) { delete s; }

void fa2_session_advance(Fa2Session *s, int iters, double *h_stats) {
    if (iters <= 0) return;
    bgl_ctx *ctx = s->g->ctx;
    DevBuf<double> st;
    if (h_stats) st.reset(ctx->alloc, 3 * (size_t)iters);
    run_iterations(*s->run, iters, h_stats ? st.p : nullptr);
    s->iters_done += iters;
    if (h_stats) {
        BGL_CUDA(cudaMemcpyAsync(h_stats, st.p, sizeof(double) * 3 * iters, cudaMemcpyDeviceToHost, ctx->stream));
        BGL_CUDA(cudaStreamSynchronize(ctx->stream));
    }
}

int64_t fa2_session_positions(Fa2Session *s, float2 *h_xy) {
    cudaStream_t st = s->g->ctx->stream;
    BGL_CUDA(cudaMemcpyAsync(h_xy, s->xy.p, sizeof(float2) * s->n, cudaMemcpyDeviceToHost, st));
    BGL_CUDA(cudaStreamSynchronize(st));
    return s->iters_done;
}

size_t fa2_session_state_bytes(const Fa2Session *s) { return sizeof(StateHeader) + 2 * sizeof(float2) * s->n; }

void fa2_session_save(Fa2Session *s, void *buf) {
    StateHeader h;
    std::memset(&h, 0, sizeof(h));
    std::memcpy(h.magic, STATE_MAGIC, 8);
    h.version = STATE_VERSION;
    h.header_bytes = (uint32_t)sizeof(StateHeader);
    h.n_nodes = s->g->n;
    h.n_undir = s->g->n_undir;
    h.comp = s->c;
    h.comp_nodes = s->n;
    h.fingerprint = s->fingerprint;
    h.iters_done = s->iters_done;
    h.params = s->p;
    h.fmm_sortskip = s->run->fmm.empty() ? -1 : fmm_sortskip(s->run->fmm[0]);
    cudaStream_t st = s->g->ctx->stream;
    BGL_CUDA(cudaMemcpyAsync(&h.sg, s->run->sg.p, sizeof(double), cudaMemcpyDeviceToHost, st));
    char *out = static_cast<char *>(buf);
    float2 *xy = reinterpret_cast<float2 *>(out + sizeof(StateHeader));
    BGL_CUDA(cudaMemcpyAsync(xy, s->xy.p, sizeof(float2) * s->n, cudaMemcpyDeviceToHost, st));
    BGL_CUDA(cudaMemcpyAsync(xy + s->n, s->run->fprev.p, sizeof(float2) * s->n, cudaMemcpyDeviceToHost, st));
    BGL_CUDA(cudaStreamSynchronize(st));
    std::memcpy(out, &h, sizeof(h));
}

Fa2Session *fa2_session_load(bgl_graph *g, const void *buf, size_t len) {
    BGL_REQUIRE(len >= sizeof(StateHeader), "state: buffer shorter than the header");
    StateHeader h;
    std::memcpy(&h, buf, sizeof(h));
    if (std::memcmp(h.magic, STATE_MAGIC, 8) != 0 || h.version != STATE_VERSION ||
        h.header_bytes != sizeof(StateHeader))
        fail(BGL_EINVAL, "state: not a ForceAtlas2 checkpoint of this library version");
    if (!g->has_comp) fail(BGL_ESTATE, "state: run bgl_components before loading a checkpoint");
    if (h.n_nodes != g->n || h.n_undir != g->n_undir || h.comp < 0 || h.comp >= g->n_comp ||
        h.comp_nodes != g->h_comp_off[h.comp + 1] - g->h_comp_off[h.comp])
        fail(BGL_EINVAL, "state: the checkpoint belongs to another graph");
    BGL_REQUIRE(len >= sizeof(StateHeader) + 2 * sizeof(float2) * (size_t)h.comp_nodes,
                "state: buffer shorter than the checkpoint");
    check_params(&h.params);
    Fa2Session *s = session_new(g, &h.params, h.comp);
    try {
        if (s->fingerprint != h.fingerprint) fail(BGL_EINVAL, "state: the checkpoint belongs to another graph");
        const float2 *xy = reinterpret_cast<const float2 *>(static_cast<const char *>(buf) + sizeof(StateHeader));
        cudaStream_t st = g->ctx->stream;
        BGL_CUDA(cudaMemcpyAsync(s->xy.p, xy, sizeof(float2) * s->n, cudaMemcpyHostToDevice, st));
        BGL_CUDA(cudaMemcpyAsync(s->run->fprev.p, xy + s->n, sizeof(float2) * s->n, cudaMemcpyHostToDevice, st));
        BGL_CUDA(cudaMemcpyAsync(s->run->sg.p, &h.sg, sizeof(double), cudaMemcpyHostToDevice, st));
        BGL_CUDA(cudaStreamSynchronize(st));
        if ((h.fmm_sortskip >= 0) != !s->run->fmm.empty()) fail(BGL_EINVAL, "state: repulsion kind mismatch");
        if (h.fmm_sortskip >= 0) fmm_set_sortskip(s->run->fmm[0], h.fmm_sortskip);
        s->iters_done = h.iters_done;
    } catch (...) {
        delete s;
        throw;
    }
    return s;
}

void fa2_forces(bgl_graph *g, const bgl_params *p, const float2 *xy, float2 *f, int64_t c, int what) {
    int64_t q0 = g->h_comp_off[c];
    Fa2Run run(g, p, const_cast<float2 *>(xy), q0, c, c + 1);
    run.forces(what);
    BGL_CUDA(cudaMemcpyAsync(f, run.f.p, sizeof(float2) * (run.q1 - run.q0), cudaMemcpyDeviceToDevice,
                             g->ctx->stream));
    BGL_CUDA(cudaStreamSynchronize(g->ctx->stream));
    run.check_fmm();
}

}  // namespace bgl
