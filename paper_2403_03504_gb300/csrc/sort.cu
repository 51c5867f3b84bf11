// Device primitives: multi-block exclusive scan and stable LSD radix sort.
//
// Scan: reduce-then-scan over tiles of 4096 elements (512 threads x 8).
// Radix sorts: 8-bit digits, tiles of 4,096 keys, a single kernel a pass
// (onesweep, below), in which each warp ranks its keys by votes on their
// digits so that equal digits keep their input order (stable).
#include <algorithm>
#include <cstdlib>

#include "bgl_internal.cuh"
#include "sort_hist.cuh"

namespace bgl {

namespace {

constexpr int SCAN_THREADS = 512;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__device__ T block_exclusive_scan(T v, T *warp_tot, T *total) {
    // exclusive scan of one value per thread across the block
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nwarps ? warp_tot[lane] : T(0);
        T s = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nwarps) warp_tot[lane] = s - w;   // exclusive warp offsets
        if (lane == nwarps - 1) *total = s;
    }
    __syncthreads();
    T r = warp_tot[warp] + x - v;
    __syncthreads();
    return r;
}

template <typename T>
__global__ void scan_reduce_kernel(const T *__restrict__ in, T *__restrict__ tile_sum, int64_t n) {
    __shared__ T red[SCAN_THREADS / 32];
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int64_t k = base + (int64_t)i * SCAN_THREADS + threadIdx.x;
        if (k < n) s += in[k];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; ++w) t += red[w];
        tile_sum[blockIdx.x] = t;
    }
}

// single block: exclusive scan of the tile sums, in place; total to *d_total
template <typename T>
__global__ void scan_tiles_kernel(T *tile_sum, int64_t ntiles, T *d_total) {
    __shared__ T wt[32];
    __shared__ T tot;
    T carry = 0;
    for (int64_t b = 0; b < ntiles; b += blockDim.x) {
        int64_t k = b + threadIdx.x;
        T v = k < ntiles ? tile_sum[k] : T(0);
        T e = block_exclusive_scan<T>(v, wt, &tot);
        if (k < ntiles) tile_sum[k] = carry + e;
        carry += tot;
        __syncthreads();
    }
    if (threadIdx.x == 0 && d_total) *d_total = carry;
}

template <typename T>
__global__ void scan_apply_kernel(const T *__restrict__ in, T *__restrict__ out, const T *__restrict__ tile_off,
                                  int64_t n) {
    __shared__ T buf[SCAN_TILE];
    __shared__ T wt[32];
    __shared__ T tot;
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int idx = i * SCAN_THREADS + threadIdx.x;
        int64_t k = base + idx;
        buf[idx] = k < n ? in[k] : T(0);
    }
    __syncthreads();
    T v[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = buf[threadIdx.x * SCAN_ITEMS + i];
        s += v[i];
    }
    T e = block_exclusive_scan<T>(s, wt, &tot) + tile_off[blockIdx.x];
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        buf[threadIdx.x * SCAN_ITEMS + i] = e;
        e += v[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        int idx = i * SCAN_THREADS + threadIdx.x;
        int64_t k = base + idx;
        if (k < n) out[k] = buf[idx];
    }
}

template <typename T>
void scan_exclusive(bgl_ctx *c, const T *in, T *out, int64_t n, T *d_total, T *tiles = nullptr) {
    if (n <= 0) {
        if (d_total) BGL_CUDA(cudaMemsetAsync(d_total, 0, sizeof(T), c->stream));
        return;
    }
    int64_t ntiles = (n + SCAN_TILE - 1) / SCAN_TILE;
    DevBuf<T> own;
    if (!tiles) {
        own.reset(c->alloc, ntiles);
        tiles = own.p;
    }
    scan_reduce_kernel<T><<<(unsigned)ntiles, SCAN_THREADS, 0, c->stream>>>(in, tiles, n);
    BGL_LAUNCH_CHECK();
    scan_tiles_kernel<T><<<1, 1024, 0, c->stream>>>(tiles, ntiles, d_total);
    BGL_LAUNCH_CHECK();
    scan_apply_kernel<T><<<(unsigned)ntiles, SCAN_THREADS, 0, c->stream>>>(in, out, tiles, n);
    BGL_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ radix sort

// ------------------------------------------------------------------ onesweep
//
// Four 8-bit digit passes.  One histogram kernel counts all four digit
// histograms at once and its last block turns them into global digit
// bases.  Each pass is then a single kernel: tiles take increasing indices
// from a ticket counter, rank their keys stably (per-warp votes on the digit and
// counts, warps in order), publish their per-digit counts, and look back
// over earlier tiles' published counts (decoupled look-back, Merrill and
// Garland) for their global offsets; keys are regrouped by digit in shared
// memory so each digit run is written with coalesced stores.  Waits are
// bounded; a wait that gives up records an error bit and the tile carries on.

// OS_THREADS, OS_ITEMS, OS_TILE: sort_hist.cuh (a caller's histogram kernel uses the same tiles)
constexpr int OS_WARPS = OS_THREADS / 32;
// A look-back word: two flag bits above the count, of 32 bits for counts
// below 2^30 and of 64 bits for more.
template <typename W>
struct OsWord {
    static constexpr W AGG = W(1) << (8 * sizeof(W) - 2), INC = W(2) << (8 * sizeof(W) - 2), MASK = AGG - 1;
};
constexpr long long OS_SPIN = 1ll << 24;
constexpr int OS_LB = 8;           // look-back window (predecessor tiles per step)

// Decoupled look-back of digit d: publishes the tile's count `own` and returns
// the sum of the earlier tiles' counts.  OS_LB predecessors per step: their
// status words are loaded together, then taken newest first until an
// inclusive one.
template <typename W>
__device__ __forceinline__ uint32_t os_look_back(volatile W *st, int tile, int d, uint32_t own, int *err,
                                                 const OsWait &wait) {
    uint32_t excl = 0;
    if (tile == 0) {
        if (!wait.stall_first) st[d] = OsWord<W>::INC | own;
        return 0;
    }
    st[(int64_t)tile * 256 + d] = OsWord<W>::AGG | own;
    bool done = false;
    for (int t = tile - 1; t >= 0 && !done; t -= OS_LB) {
        W v[OS_LB];
#pragma unroll
        for (int w = 0; w < OS_LB; ++w) v[w] = t - w >= 0 ? (W)st[(int64_t)(t - w) * 256 + d] : OsWord<W>::INC;
#pragma unroll
        for (int w = 0; w < OS_LB; ++w) {
            if (done) break;
            long long it = 0;
            while ((v[w] & ~OsWord<W>::MASK) == 0) {
                if (++it > wait.spin) {
                    atomicOr(err, 1);
                    v[w] = OsWord<W>::INC;
                    break;
                }
                __nanosleep(32);
                v[w] = st[(int64_t)(t - w) * 256 + d];
            }
            excl += (uint32_t)(v[w] & OsWord<W>::MASK);
            if (v[w] & OsWord<W>::INC) done = true;
        }
    }
    __threadfence();
    st[(int64_t)tile * 256 + d] = OsWord<W>::INC | (excl + own);
    return excl;
}

// Buffers of pass d (0..3) when the first `skip` passes are skipped: the
// first active pass reads the input, the last writes the output, the ones
// between alternate between the two scratch pairs.
struct OsBufs {
    uint32_t *keys, *vals;      // input, and output of the last pass
    uint32_t *k0, *v0, *k1, *v1; // scratch
};

__global__ void __launch_bounds__(OS_THREADS, 2) os_scatter_kernel(OsBufs bf, int d, const int *d_skip, int64_t n,
                                                                   const uint32_t *__restrict__ base,
                                                                   uint32_t *status, unsigned *ticket, int *err,
                                                                   const float2 *__restrict__ gxy,
                                                                   const float *__restrict__ gmass,
                                                                   float4 *__restrict__ gpts, OsWait wait) {
    const int skip = d_skip ? *d_skip : 0;
    if (d < skip) return;
    const int shift = 8 * d;
    const uint32_t *__restrict__ kin = d == skip ? bf.keys : (((d - skip - 1) & 1) ? bf.k1 : bf.k0);
    const uint32_t *__restrict__ vin = d == skip ? bf.vals : (((d - skip - 1) & 1) ? bf.v1 : bf.v0);
    uint32_t *__restrict__ kout = d == 3 ? bf.keys : (((d - skip) & 1) ? bf.k1 : bf.k0);
    uint32_t *__restrict__ vout = d == 3 ? bf.vals : (((d - skip) & 1) ? bf.v1 : bf.v0);
    __shared__ __align__(4) uint16_t cnt[OS_WARPS][256];     // (at most a tile)
    __shared__ uint32_t gofs[256];
    __shared__ int32_t lstart[256];
    __shared__ int32_t wsum[8];
    __shared__ uint32_t skey[OS_TILE], sval[OS_TILE];
    __shared__ int tile_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // after a wait gave up (in an earlier pass, or in this one before the
    // block started) the keys are not sorted: blocks return before taking
    // a tile, so no tile is left waiting for one that nobody holds
    if (threadIdx.x == 0) tile_s = (*(volatile int *)err & 1) ? -1 : (int)atomicAdd(ticket, 1u);
    for (int i = threadIdx.x; i < OS_WARPS * 128; i += OS_THREADS) reinterpret_cast<uint32_t *>(cnt)[i] = 0;
    __syncthreads();
    const int tile = tile_s;
    if (tile < 0) return;
    const int64_t t0 = (int64_t)tile * OS_TILE;
    const int tcount = (int)(n - t0 < OS_TILE ? n - t0 : OS_TILE);
    const unsigned lt = (1u << lane) - 1u;
    const int64_t wbase = t0 + (int64_t)warp * 32 * OS_ITEMS;
    uint32_t key[OS_ITEMS], val[OS_ITEMS];
    int32_t rank[OS_ITEMS];
    // all loads in flight before the ranking (whose warp barriers would
    // otherwise order them one after another)
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int64_t k = wbase + r * 32 + lane;
        key[r] = k < n ? kin[k] : 0u;
        val[r] = k < n ? vin[k] : 0u;
    }
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int64_t k = wbase + r * 32 + lane;
        const bool ok = k < n;
        const unsigned d = (key[r] >> shift) & 0xFF;
        const unsigned peers = digit_peers(d, ok);
        const int before = __popc(peers & lt);
        const int cur = ok ? cnt[warp][d] : 0;
        __syncwarp();
        if (ok && before == 0) cnt[warp][d] = (uint16_t)(cur + __popc(peers));
        __syncwarp();
        rank[r] = ok ? cur + before : -1;
    }
    __syncthreads();
    // thread = digit: prefix over warps, then an exclusive scan over digits
    // (tile-local start of each digit run), then the look-back for the
    // global offset of each digit run
    const bool digit = threadIdx.x < 256;
    int s = 0, x = 0;
    if (digit) {
        const int d = threadIdx.x;
#pragma unroll
        for (int w = 0; w < OS_WARPS; ++w) {
            const int c = cnt[w][d];
            cnt[w][d] = (uint16_t)s;
            s += c;
        }
        x = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        const uint32_t excl = os_look_back<uint32_t>(status, tile, d, (uint32_t)s, err, wait);
        gofs[d] = base[d] + excl;
    }
    __syncthreads();
    if (digit) {
        int pre = 0;
        for (int w = 0; w < warp; ++w) pre += wsum[w];
        lstart[threadIdx.x] = pre + x - s;
    }
    __syncthreads();
    // keys to their tile-local sorted position, then coalesced runs to global
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        if (rank[r] < 0) continue;
        const unsigned d = (key[r] >> shift) & 0xFF;
        const int lp = lstart[d] + cnt[warp][d] + rank[r];
        skey[lp] = key[r];
        sval[lp] = val[r];
    }
    __syncthreads();
    uint32_t dst[OS_ITEMS];
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int i = r * OS_THREADS + threadIdx.x;
        key[r] = i < tcount ? skey[i] : 0u;
        val[r] = i < tcount ? sval[i] : 0u;
        const unsigned d = (key[r] >> shift) & 0xFF;
        dst[r] = gofs[d] + (uint32_t)(i - lstart[d]);
    }
    if (gpts) {
        // last pass with a gather: the sorted record {x, y, m, index}, all
        // gather loads issued before the stores
        float2 p[OS_ITEMS];
        float m[OS_ITEMS];
#pragma unroll
        for (int r = 0; r < OS_ITEMS; ++r) {
            const bool ok = r * OS_THREADS + (int)threadIdx.x < tcount;
            p[r] = ok ? gxy[val[r]] : make_float2(0.f, 0.f);
            m[r] = ok ? gmass[val[r]] : 0.f;
        }
#pragma unroll
        for (int r = 0; r < OS_ITEMS; ++r) {
            if (r * OS_THREADS + (int)threadIdx.x >= tcount) continue;
            kout[dst[r]] = key[r];
            gpts[dst[r]] = make_float4(p[r].x, p[r].y, m[r], __int_as_float((int)val[r]));
        }
    } else {
#pragma unroll
        for (int r = 0; r < OS_ITEMS; ++r) {
            if (r * OS_THREADS + (int)threadIdx.x >= tcount) continue;
            kout[dst[r]] = key[r];
            vout[dst[r]] = val[r];
        }
    }
}

// The sort of the graph build: keys of 32 or 64 bits, with values or without,
// any number of passes.  One kernel counts the digits of every pass, one
// kernel a pass moves the keys.  A digit count, a scan of the tiles' counts in
// three kernels and a scatter took 46 us a pass for 800,000 64-bit keys with
// values and 60 for 1,600,000 without; a pass takes 18 and 25.
template <typename K>
__global__ void __launch_bounds__(OS_THREADS) sweep_hist_kernel(const K *__restrict__ keys, int64_t n, int passes,
                                                               uint32_t *hist, uint32_t *base, unsigned *counter) {
    __shared__ uint32_t sh[sizeof(K)][256];
    __shared__ uint32_t ws[OS_THREADS / 32];
    __shared__ bool last;
    for (int i = threadIdx.x; i < passes * 256; i += OS_THREADS) (&sh[0][0])[i] = 0;
    __syncthreads();
    const int64_t i0 = (int64_t)blockIdx.x * OS_TILE + threadIdx.x;
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int64_t i = i0 + (int64_t)r * OS_THREADS;
        if (i >= n) break;
        const K k = keys[i];
        for (int d = 0; d < passes; ++d) atomicAdd(&sh[d][(unsigned)(k >> (8 * d)) & 0xFFu], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += OS_THREADS)
        if ((&sh[0][0])[i]) atomicAdd(&hist[i], (&sh[0][0])[i]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i0b = 0; i0b < passes * 256; i0b += OS_THREADS) {
        const int i = i0b + threadIdx.x;
        const uint32_t v = i < passes * 256 ? __ldcg(&hist[i]) : 0u;
        uint32_t x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) ws[warp] = x;
        __syncthreads();
        uint32_t pre = 0;
        for (int w = warp & ~7; w < warp; ++w) pre += ws[w];
        if (i < passes * 256) base[i] = pre + x - v;
        __syncthreads();
    }
}

template <typename K, bool VALS, typename W>
__global__ void __launch_bounds__(OS_THREADS, 2) sweep_kernel(const K *__restrict__ kin,
                                                              const uint32_t *__restrict__ vin, K *__restrict__ kout,
                                                              uint32_t *__restrict__ vout, int64_t n, int shift,
                                                              const uint32_t *__restrict__ base, W *status,
                                                              unsigned *ticket, int *err, OsWait wait) {
    __shared__ __align__(4) uint16_t cnt[OS_WARPS][256];
    __shared__ uint32_t gofs[256];
    __shared__ int32_t lstart[256];
    __shared__ int32_t wsum[8];
    __shared__ K skey[OS_TILE];
    __shared__ int tile_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) tile_s = (*(volatile int *)err & 1) ? -1 : (int)atomicAdd(ticket, 1u);
    for (int i = threadIdx.x; i < OS_WARPS * 128; i += OS_THREADS) reinterpret_cast<uint32_t *>(cnt)[i] = 0;
    __syncthreads();
    const int tile = tile_s;
    if (tile < 0) return;              // a wait gave up: see os_scatter_kernel
    const int64_t t0 = (int64_t)tile * OS_TILE;
    const int tcount = (int)(n - t0 < OS_TILE ? n - t0 : OS_TILE);
    const unsigned lt = (1u << lane) - 1u;
    const int w0 = warp * 32 * OS_ITEMS;
    K key[OS_ITEMS];
    uint32_t val[OS_ITEMS];
    int32_t rank[OS_ITEMS];
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int i = w0 + r * 32 + lane;
        key[r] = i < tcount ? kin[t0 + i] : K(0);
        val[r] = VALS && i < tcount ? vin[t0 + i] : 0u;
    }
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const bool ok = w0 + r * 32 + lane < tcount;
        const unsigned d = (unsigned)(key[r] >> shift) & 0xFFu;
        const unsigned peers = digit_peers(d, ok);
        const int before = __popc(peers & lt);
        const int cur = ok ? cnt[warp][d] : 0;
        __syncwarp();
        if (ok && before == 0) cnt[warp][d] = (uint16_t)(cur + __popc(peers));
        __syncwarp();
        rank[r] = ok ? cur + before : -1;
    }
    __syncthreads();
    const bool digit = threadIdx.x < 256;
    int s = 0, x = 0;
    if (digit) {
        const int d = threadIdx.x;
#pragma unroll
        for (int w = 0; w < OS_WARPS; ++w) {
            const int c = cnt[w][d];
            cnt[w][d] = (uint16_t)s;
            s += c;
        }
        x = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        gofs[d] = base[d] + os_look_back<W>(status, tile, d, (uint32_t)s, err, wait);
    }
    __syncthreads();
    if (digit) {
        int pre = 0;
        for (int w = 0; w < warp; ++w) pre += wsum[w];
        lstart[threadIdx.x] = pre + x - s;
    }
    __syncthreads();
    // keys to their tile-local sorted position, then coalesced runs to
    // global; the values the same way through the same memory
    int lp[OS_ITEMS];
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const unsigned d = (unsigned)(key[r] >> shift) & 0xFFu;
        lp[r] = lstart[d] + cnt[warp][d] + rank[r];
        if (rank[r] >= 0) skey[lp[r]] = key[r];
    }
    __syncthreads();
    uint32_t dst[OS_ITEMS];
#pragma unroll
    for (int r = 0; r < OS_ITEMS; ++r) {
        const int i = r * OS_THREADS + threadIdx.x;
        const K k = i < tcount ? skey[i] : K(0);
        const unsigned d = (unsigned)(k >> shift) & 0xFFu;
        dst[r] = gofs[d] + (uint32_t)(i - lstart[d]);
        if (i < tcount) kout[dst[r]] = k;
    }
    if constexpr (VALS) {
        uint32_t *sval = reinterpret_cast<uint32_t *>(skey);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < OS_ITEMS; ++r)
            if (rank[r] >= 0) sval[lp[r]] = val[r];
        __syncthreads();
#pragma unroll
        for (int r = 0; r < OS_ITEMS; ++r) {
            const int i = r * OS_THREADS + threadIdx.x;
            if (i < tcount) vout[dst[r]] = sval[i];
        }
    }
}

inline int64_t os_tiles(int64_t n) { return (n + OS_TILE - 1) / OS_TILE; }

// Sorts in place on bits [0, bits), look-back words of type W.  A wait that
// gives up sets the context's d_flag[3], which sort_check reports.
template <typename K, bool VALS, typename W>
void radix_sort_words(bgl_ctx *c, K *keys, uint32_t *vals, int64_t n, int bits) {
    const int64_t nt = os_tiles(n);
    const int passes = (bits + 7) / 8;
    DevBuf<K> kt(c->alloc, n);
    DevBuf<uint32_t> vt;
    if (VALS) vt.reset(c->alloc, n);
    // digit counts, pass tickets and arrival counter (zero at first), digit bases
    const size_t counts = (size_t)passes * 256;
    DevBuf<uint32_t> ws(c->alloc, counts + 16), base(c->alloc, counts);
    BGL_CUDA(cudaMemsetAsync(ws.p, 0, ws.bytes(), c->stream));
    unsigned *tickets = ws.p + counts;
    // look-back words, zero before their pass: for every pass, or for many tiles one set for all
    const bool each = nt > 16384;
    DevBuf<W> status(c->alloc, 256 * (size_t)nt * (each ? 1 : passes));
    if (!each) BGL_CUDA(cudaMemsetAsync(status.p, 0, status.bytes(), c->stream));
    sweep_hist_kernel<K><<<(unsigned)nt, OS_THREADS, 0, c->stream>>>(keys, n, passes, ws.p, base.p, tickets + 15);
    BGL_LAUNCH_CHECK();
    if (nt > 1) c->sort_waits = true;      // (one tile waits for nobody)
    const OsWait wait = sort_wait(c->d_flag + 3);
    K *ka = keys, *kb = kt.p;
    uint32_t *va = vals, *vb = vt.p;
    for (int d = 0; d < passes; ++d) {
        if (each) BGL_CUDA(cudaMemsetAsync(status.p, 0, status.bytes(), c->stream));
        sweep_kernel<K, VALS, W><<<(unsigned)nt, OS_THREADS, 0, c->stream>>>(
            ka, va, kb, vb, n, 8 * d, base.p + 256 * d, status.p + (each ? 0 : (size_t)d * 256 * nt), tickets + d,
            wait.err, wait);
        BGL_LAUNCH_CHECK();
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    if (passes & 1) {
        BGL_CUDA(cudaMemcpyAsync(keys, ka, sizeof(K) * n, cudaMemcpyDeviceToDevice, c->stream));
        if (VALS) BGL_CUDA(cudaMemcpyAsync(vals, va, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, c->stream));
    }
}

template <typename K, bool VALS>
void radix_sort(bgl_ctx *c, K *keys, uint32_t *vals, int64_t n, int bits) {
    if (n <= 1 || bits <= 0) return;
    BGL_REQUIRE(n < (int64_t(1) << 31), "radix sort: more than 2^31 keys");
    if (n < (int64_t(1) << 30)) radix_sort_words<K, VALS, uint32_t>(c, keys, vals, n, bits);
    else radix_sort_words<K, VALS, unsigned long long>(c, keys, vals, n, bits);
}

}  // namespace

void scan_exclusive_i64(bgl_ctx *c, const int64_t *in, int64_t *out, int64_t n, int64_t *d_total) {
    scan_exclusive<int64_t>(c, in, out, n, d_total);
}
void scan_exclusive_i32(bgl_ctx *c, const int32_t *in, int32_t *out, int64_t n, int32_t *d_total) {
    scan_exclusive<int32_t>(c, in, out, n, d_total);
}
void radix_sort_u64(bgl_ctx *c, uint64_t *keys, uint32_t *vals, int64_t n, int bits) {
    if (vals) radix_sort<uint64_t, true>(c, keys, vals, n, bits);
    else radix_sort<uint64_t, false>(c, keys, nullptr, n, bits);
}
void radix_sort_u32(bgl_ctx *c, uint32_t *keys, uint32_t *vals, int64_t n, int bits) {
    if (vals) radix_sort<uint32_t, true>(c, keys, vals, n, bits);
    else radix_sort<uint32_t, false>(c, keys, nullptr, n, bits);
}
OsWait sort_wait(int *err) {
    OsWait w;
    w.err = err;
    w.spin = OS_SPIN;
    const char *v = std::getenv("BGL_TEST_SORT_STALL");
    if (v && v[0] == '1') {
        w.stall_first = 1;
        w.spin = 1 << 12;
    }
    return w;
}
void sort_fetch(bgl_ctx *c) {
    if (c->sort_waits)
        BGL_CUDA(cudaMemcpyAsync(c->h_flag + 3, c->d_flag + 3, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
}
void sort_fetched(bgl_ctx *c) {
    if (!c->sort_waits) return;
    c->sort_waits = false;
    if (!c->h_flag[3]) return;
    c->h_flag[3] = 0;
    BGL_CUDA(cudaMemsetAsync(c->d_flag + 3, 0, sizeof(int), c->stream));
    fail(BGL_ETIMEOUT, "radix sort: a bounded device-side wait gave up");
}
void sort_check(bgl_ctx *c) {
    if (!c->sort_waits) return;
    sort_fetch(c);
    BGL_CUDA(cudaStreamSynchronize(c->stream));
    sort_fetched(c);
}

void SortWorkspace::reserve(Allocator *a, int64_t n, cudaStream_t s) {
    if (n <= cap) return;
    cap = 0;
    keys.reset(a, n);
    vals.reset(a, n);
    keys2.reset(a, n);
    vals2.reset(a, n);
    // hist: 4 x 256 digit counts, 4 x 256 digit bases, 4 tickets, 1 counter
    hist.reset(a, 8 * 256 + 5);
    BGL_CUDA(cudaMemsetAsync(hist.p, 0, hist.bytes(), s));
    tiles.reset(a, 4 * 256 * os_tiles(n));   // look-back status words, one block per pass
    cap = n;
}

OsHist radix_sort_u32_ws_begin(SortWorkspace &ws, int64_t n) {
    BGL_REQUIRE(n <= ws.cap && n < (int64_t(1) << 30), "radix sort: workspace too small");
    OsHist h;
    h.hist = reinterpret_cast<uint32_t *>(ws.hist.p);
    h.base = h.hist + 4 * 256;
    unsigned *tickets = reinterpret_cast<unsigned *>(h.hist + 8 * 256);
    h.counter = tickets + 4;
    h.tickets = tickets;
    h.status = reinterpret_cast<uint32_t *>(ws.tiles.p);
    h.ntiles = os_tiles(n);
    return h;
}

void radix_sort_u32_ws_scatter(bgl_ctx *c, SortWorkspace &ws, uint32_t *keys, uint32_t *vals, int64_t n,
                               const float2 *gxy, const float *gmass, float4 *gpts, const int *d_skip,
                               const OsWait &wait) {
    BGL_REQUIRE(wait.err && wait.spin > 0, "radix sort: waits without a bound or a word for their failure");
    cudaStream_t s = c->stream;
    const int64_t nt = os_tiles(n);
    uint32_t *hist = reinterpret_cast<uint32_t *>(ws.hist.p);
    uint32_t *base = hist + 4 * 256;
    unsigned *tickets = reinterpret_cast<unsigned *>(hist + 8 * 256);
    uint32_t *status = reinterpret_cast<uint32_t *>(ws.tiles.p);
    const OsBufs bf{keys, vals, ws.keys.p, ws.vals.p, ws.keys2.p, ws.vals2.p};
    for (int d = 0; d < 4; ++d) {
        const bool g = d == 3 && gpts;
        os_scatter_kernel<<<(unsigned)nt, OS_THREADS, 0, s>>>(bf, d, d_skip, n, base + 256 * d,
                                                              status + (int64_t)d * 256 * nt, tickets + d, wait.err,
                                                              g ? gxy : nullptr, g ? gmass : nullptr,
                                                              g ? gpts : nullptr, wait);
        BGL_LAUNCH_CHECK();
    }
    // the sorted keys (and values unless gathered) are back in keys / vals
}

int bits_for(uint64_t v) {
    int b = 0;
    while (b < 64 && (v >> b) != 0) ++b;
    return b;
}

}  // namespace bgl
