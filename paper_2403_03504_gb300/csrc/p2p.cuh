// Pair kernel of the direct repulsion sum (Section 3.2), shared by the
// exact comparator and the near field of the FMM.
#pragma once

namespace bgl {

__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// One pair of the direct sum: f += m_j (z - z_j) / (|z - z_j|^2 + 1e-30) for
// the target (zx, zy) and the source q = (x_j, y_j, m_j, .).  A coincident
// pair (the target itself) has dx = dy = 0 and adds exactly 0; for any other
// pair of FP32 points the 1e-30 shift is far below one rounding of r^2.
// Costs 7 FP32 operations and one MUFU reciprocal.
__device__ __forceinline__ void p2p_pair(float zx, float zy, const float4 &q, float &fx, float &fy) {
    const float dx = zx - q.x, dy = zy - q.y;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, 1e-30f));
    const float w = q.z * rcp_approx(r2);
    fx = fmaf(w, dx, fx);
    fy = fmaf(w, dy, fy);
}

// Two targets against one source with the packed FP32x2 instructions of
// sm_100 and later (one issue slot for two lanes' worth of add, multiply or
// FMA): 7 packed operations and two reciprocals for two pairs.  The targets
// come negated (nzx = -zx) and the accumulators hold the negated sums,
// g += m_j (z_j - z) / (|z_j - z|^2 + 1e-30): each operation is the sign
// mirror of p2p_pair's (round-to-nearest is symmetric in sign), so -g equals,
// bit for bit, what p2p_pair accumulates in the same order.
__device__ __forceinline__ void p2p_pair2(float2 nzx, float2 nzy, const float4 &q, float2 &gx, float2 &gy) {
    const float2 dx = __fadd2_rn(make_float2(q.x, q.x), nzx);
    const float2 dy = __fadd2_rn(make_float2(q.y, q.y), nzy);
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, make_float2(1e-30f, 1e-30f)));
    const float2 w = __fmul2_rn(make_float2(q.z, q.z), make_float2(rcp_approx(r2.x), rcp_approx(r2.y)));
    gx = __ffma2_rn(w, dx, gx);
    gy = __ffma2_rn(w, dy, gy);
}

// Sources a warp takes together in p2p_chain; src holds this many readable
// entries past the last source.
constexpr int P2P_AHEAD = 8;

// f += the pairs of one target with src[0 .. cnt) in order, for a warp that
// has its scheduler to itself: the terms of eight sources are worked out
// (their reciprocals in flight together, the next eight sources loading)
// while those of the eight before are added, so that neither the MUFU's
// latency nor the chain of additions is waited for.  Bit for bit the sums of
// p2p_pair in a loop.  r2_of(dx, dy) is the guarded squared distance.
template <class R2>
__device__ __forceinline__ void p2p_chain(float zx, float zy, const float4 *src, int cnt, R2 r2_of, float &fx,
                                          float &fy) {
    constexpr int B = P2P_AHEAD;
    const int full = cnt / B;
    if (full > 0) {
        float4 q[B];
        float dx[B], dy[B], w[B];
#pragma unroll
        for (int k = 0; k < B; ++k) q[k] = src[k];
#pragma unroll
        for (int k = 0; k < B; ++k) {
            dx[k] = zx - q[k].x;
            dy[k] = zy - q[k].y;
            w[k] = q[k].z * rcp_approx(r2_of(dx[k], dy[k]));
        }
#pragma unroll
        for (int k = 0; k < B; ++k) q[k] = src[B + k];
#pragma unroll 2
        for (int b = 1; b < full; ++b) {
            const float4 *next = src + (b + 1) * B;
            float ex[B], ey[B], v[B];
#pragma unroll
            for (int k = 0; k < B; ++k) {
                ex[k] = zx - q[k].x;
                ey[k] = zy - q[k].y;
                v[k] = q[k].z * rcp_approx(r2_of(ex[k], ey[k]));
                q[k] = next[k];
                fx = fmaf(w[k], dx[k], fx);
                fy = fmaf(w[k], dy[k], fy);
            }
#pragma unroll
            for (int k = 0; k < B; ++k) {
                dx[k] = ex[k];
                dy[k] = ey[k];
                w[k] = v[k];
            }
        }
#pragma unroll
        for (int k = 0; k < B; ++k) {
            fx = fmaf(w[k], dx[k], fx);
            fy = fmaf(w[k], dy[k], fy);
        }
    }
    for (int j = full * B; j < cnt; ++j) {
        const float4 q = src[j];
        const float dx = zx - q.x, dy = zy - q.y;
        const float w = q.z * rcp_approx(r2_of(dx, dy));
        fx = fmaf(w, dx, fx);
        fy = fmaf(w, dy, fy);
    }
}

}  // namespace bgl
