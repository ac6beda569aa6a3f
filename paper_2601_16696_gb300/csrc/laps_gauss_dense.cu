// laps_gauss_dense.cu -- log p and gradient of a Gaussian given by a dense
// precision matrix P (the rotated ill-conditioned Gaussian of the paper's
// Sec. 6):  log p = -1/2 x^T P x,  grad log p = -P x,  for the ensemble's
// points as one chains-by-coordinates contraction G = -W P.
//
// A block owns a few chains per warp (CW x warps, launch_q): their points stay in
// shared memory as pairs (x_k, x_k), P streams through shared memory kRows rows at a
// time (two buffers, cp.async), and lane l of the chain's warp accumulates the column
// pairs 2 l + 64 p in packed arithmetic.
//
// The target is ill-conditioned (condition number ~1e5 in the paper's
// experiment), so -P x cancels: a binary32 dot product loses ~1e-4 of max|g|.
// The sums run in the biased form of laps_resident.cuh (dense_bias_add: four
// operations per product); a chain whose result is too small against its bias for
// that form's accuracy (dense_bias_ok) is recomputed in the compensated form, in a
// second pass of its block.  log p sums x_o (P x)_o compensated, one warp butterfly
// per chain.
//
// Bound by the FMA pipe (4 M d d_pad operations) and the operand loads: M = 1500,
// d = 300 takes 38 us, 91 us before (scalar compensated sums of ten operations a
// product, 188 blocks on 152 SMs).
#include <cuda_runtime.h>

#include <algorithm>

#include "laps_internal.h"

namespace laps {

namespace {
constexpr int kRows = 16;       // rows of P per chunk (d_pad is a multiple of 32)
constexpr int kMaxWarps = 16;

// W [M][dp] points (zero padded), P [dp][dp] symmetric (zero padded) and its row norms
// [dp], dp = 32 Q.  G [M][dp] receives -P x (zeros in the padding), LP [M] log p as
// float-float.  nw: warps that hold chains (the block's other warps only stage).
template <int Q, int CW>
__global__ void __launch_bounds__(32 * kMaxWarps) gauss_dense_grad_kernel(const float* __restrict__ P, int d,
                                                                     const float* __restrict__ W, int64_t M, int nw,
                                                                     float* __restrict__ G,
                                                                     float2* __restrict__ LP,
                                                                     const int* __restrict__ guard) {
    if (guard != nullptr && *guard == 0) return;  // the iteration no longer runs
    constexpr int dp = 32 * Q, NP = (Q + 1) / 2;
    extern __shared__ __align__(16) float sm[];
    const int nch = nw * CW;
    float* Xs = sm;                    // [nch][2 dp] pairs
    float* Ps = sm + nch * 2 * dp;     // [2][kRows][dp]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthr = blockDim.x;
    const int64_t m0 = (int64_t)blockIdx.x * nch;
    const int nc = (int)(M - m0 < nch ? M - m0 : nch);
    auto stage = [&](int k0, int buf) {  // rows k0 .. k0 + kRows - 1 of P, one commit group
        const float* src = P + (size_t)k0 * dp;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Ps + buf * kRows * dp);
        for (int o = tid; o < kRows * dp / 4; o += nthr)
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * o), "l"(src + 4 * o) : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage(0, 0);
    for (int o = tid; o < nch * dp / 4; o += nthr) {
        const int c = o / (dp / 4), j = o - c * (dp / 4);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (c < nc) v = reinterpret_cast<const float4*>(W + (m0 + c) * dp)[j];
        float4* dst = reinterpret_cast<float4*>(Xs + c * 2 * dp + 8 * j);
        dst[0] = make_float4(v.x, v.x, v.y, v.y);
        dst[1] = make_float4(v.z, v.z, v.w, v.w);
    }
    __syncthreads();  // the points are staged
    const int ch0 = CW * warp;           // this warp's first chain (warp < nw)
    const bool work = warp < nw;
    const bool tail = Q % 2 == 0 || lane < 16;  // odd Q: the last pair exists for 16 lanes
    // one pass over P's rows: row(kk, x pairs of two rows per chain offset, chunk)
    auto stream = [&](auto&& body) {
        for (int k0 = 0, b = 0; k0 < d; k0 += kRows, b ^= 1) {
            if (k0 + kRows < d) {
                stage(k0 + kRows, b ^ 1);
                asm volatile("cp.async.wait_group 1;" ::: "memory");
            } else {
                asm volatile("cp.async.wait_group 0;" ::: "memory");
            }
            __syncthreads();
            // rows past d of P are zero: they would add exact zeros, so stop at d (rounded up to 2)
            const int kn = d - k0 < kRows ? d - k0 : kRows;
            if (work) body(k0, kn, Ps + b * kRows * dp + 2 * lane);
            __syncthreads();  // the buffer may be overwritten
        }
    };
    // -P x of one chain and its log p
    auto finish = [&](int ch, const float (&r)[2 * NP]) {
        ff l = ff_make(0.0f);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            if (p == NP - 1 && !tail) continue;
            const int o = 2 * lane + 64 * p;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float xo = Xs[ch * 2 * dp + 2 * (o + e)], rv = r[2 * p + e];
                const float pr = xo * rv;
                l = ff_add(l, ff{pr, fmaf(xo, rv, -pr)});
            }
            if (ch < nc)
                *reinterpret_cast<float2*>(G + (m0 + ch) * dp + o) =
                    make_float2(o < d ? -r[2 * p] : 0.0f, o + 1 < d ? -r[2 * p + 1] : 0.0f);
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const ff w{__shfl_xor_sync(0xffffffffu, l.hi, off), __shfl_xor_sync(0xffffffffu, l.lo, off)};
            l = ff_add(l, w);
        }
        if (lane == 0 && ch < nc) LP[m0 + ch] = make_float2(-0.5f * l.hi, -0.5f * l.lo);
    };

    f32x2 S[CW][NP], lo[CW][NP];
    float nx[CW];
    const float2* sn = reinterpret_cast<const float2*>(P + (size_t)dp * dp) + lane;
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        float n2 = 0.0f;
        if (work)
            for (int o = lane; o < d; o += 32) n2 = fmaf(Xs[(ch0 + c) * 2 * dp + 2 * o], Xs[(ch0 + c) * 2 * dp + 2 * o], n2);
        nx[c] = sqrtf(group_sum<32>(n2));
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float2 np = p < NP - 1 || tail ? sn[32 * p] : make_float2(0.0f, 0.0f);
            S[c][p] = pack2(dense_sigma(nx[c], np.x), dense_sigma(nx[c], np.y));
            lo[c][p] = 0;
        }
    }
    const f32x2 m1 = pack2(-1.0f, -1.0f);
    stream([&](int k0, int kn, const float* Pc) {
#pragma unroll 2
        for (int kk = 0; kk < kn; kk += 2) {
            ulonglong2 xx[CW];
#pragma unroll
            for (int c = 0; c < CW; ++c) xx[c] = *reinterpret_cast<const ulonglong2*>(Xs + (ch0 + c) * 2 * dp + 2 * (k0 + kk));
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                f32x2 p0 = 0, p1 = 0;
                if (p < NP - 1 || tail) {
                    p0 = *reinterpret_cast<const f32x2*>(Pc + kk * dp + 64 * p);
                    p1 = *reinterpret_cast<const f32x2*>(Pc + (kk + 1) * dp + 64 * p);
                }
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    dense_bias_add(xx[c].x, p0, m1, S[c][p], lo[c][p]);
                    dense_bias_add(xx[c].y, p1, m1, S[c][p], lo[c][p]);
                }
            }
        }
    });
    unsigned again = 0u;  // bit c: chain c of this warp needs the compensated form
    if (work) {
#pragma unroll
        for (int c = 0; c < CW; ++c) {
            float r[2 * NP], rmax = 0.0f, smax = 0.0f;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const float2 np = p < NP - 1 || tail ? sn[32 * p] : make_float2(0.0f, 0.0f);
                const float s0 = dense_sigma(nx[c], np.x), s1 = dense_sigma(nx[c], np.y);
                const float2 Sv = unpack2(S[c][p]), lv = unpack2(lo[c][p]);
                r[2 * p] = (Sv.x - s0) + lv.x;
                r[2 * p + 1] = (Sv.y - s1) + lv.y;
                rmax = fmaxf(rmax, fmaxf(fabsf(r[2 * p]), fabsf(r[2 * p + 1])));
                smax = fmaxf(smax, fmaxf(s0, s1));
            }
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, off));
                smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, off));
            }
            if ((!dense_bias_ok(rmax, smax) || !(nx[c] < 3e38f)) && ch0 + c < nc) {
                bool nz = false;  // x = 0 needs no repeat: its r is exactly 0
                for (int o = lane; o < d; o += 32) nz = nz || Xs[(ch0 + c) * 2 * dp + 2 * o] != 0.0f;
                if (__any_sync(0xffffffffu, nz)) again |= 1u << c;
            }
            finish(ch0 + c, r);
        }
    }
    if (!__syncthreads_or((int)again)) return;
    for (int c = 0; c < CW; ++c) {  // rare: another pass of the block per chain slot
        stage(0, 0);
        float hi[2 * NP], lw[2 * NP];
#pragma unroll
        for (int q = 0; q < 2 * NP; ++q) hi[q] = lw[q] = 0.0f;
        stream([&](int k0, int kn, const float* Pc) {
            for (int kk = 0; kk < kn; ++kk) {
                const float x = Xs[(ch0 + c) * 2 * dp + 2 * (k0 + kk)];
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    if (p == NP - 1 && !tail) continue;
                    const float2 pv = *reinterpret_cast<const float2*>(Pc + kk * dp + 64 * p);
                    dense_comp_add(x, pv.x, hi[2 * p], lw[2 * p]);
                    dense_comp_add(x, pv.y, hi[2 * p + 1], lw[2 * p + 1]);
                }
            }
        });
        if ((again >> c) & 1u) {
#pragma unroll
            for (int q = 0; q < 2 * NP; ++q) hi[q] += lw[q];
            finish(ch0 + c, hi);
        }
    }
}

// |P_i| of every row (and, P being symmetric, column), one warp per row
__global__ void dense_row_norms_kernel(float* __restrict__ P, int dp) {
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= dp) return;
    float a = 0.0f;
    for (int j = lane; j < dp; j += 32) a = fmaf(P[(size_t)i * dp + j], P[(size_t)i * dp + j], a);
    a = group_sum<32>(a);
    if (lane == 0) P[(size_t)dp * dp + i] = sqrtf(a);
}

// Chains per block: an SM holds one block, so the ensemble is split evenly over the
// SMs (M = 1500: ten chains a block, 150 blocks; eight a block were 188 blocks, of
// which 36 SMs held two).  A warp takes one chain while 16 warps hold the block's,
// else two or (while the accumulators' 4 CW NP registers allow) four, and more than
// that runs in equal waves.
template <int Q, int CW>
cudaError_t launch_cw(const float* P, int d, const float* W, int64_t M, int per_sm, float* G, float2* LP,
                      cudaStream_t st, const int* guard) {
    const int waves = (per_sm + CW * kMaxWarps - 1) / (CW * kMaxWarps);
    const int nw = (per_sm + CW * waves - 1) / (CW * waves), nch = nw * CW;
    const size_t smem = (size_t)(2 * nch + 2 * kRows) * 32 * Q * sizeof(float);
    cudaError_t e = ensure_dyn_smem((const void*)gauss_dense_grad_kernel<Q, CW>, smem);
    if (e != cudaSuccess) return e;
    const int64_t blocks = (M + nch - 1) / nch;
    gauss_dense_grad_kernel<Q, CW><<<(unsigned)blocks, 32 * std::max(nw, 4), smem, st>>>(P, d, W, M, nw, G, LP, guard);
    return cudaGetLastError();
}
template <int Q>
cudaError_t launch_q(const float* P, int d, const float* W, int64_t M, float* G, float2* LP, cudaStream_t st,
                     const int* guard) {
    int dev = 0, nsm = 1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int per_sm = (int)std::min<int64_t>((M + nsm - 1) / nsm, 1 << 20);
    if (per_sm <= kMaxWarps) return launch_cw<Q, 1>(P, d, W, M, per_sm, G, LP, st, guard);
    if constexpr (Q <= 8)
        if (per_sm > 2 * kMaxWarps) return launch_cw<Q, 4>(P, d, W, M, per_sm, G, LP, st, guard);
    return launch_cw<Q, 2>(P, d, W, M, per_sm, G, LP, st, guard);
}
}  // namespace

cudaError_t dense_row_norms(float* P, int d_pad, cudaStream_t st) {
    dense_row_norms_kernel<<<(d_pad * 32 + 255) / 256, 256, 0, st>>>(P, d_pad);
    return cudaGetLastError();
}

cudaError_t gauss_dense_grad(const float* P, int d_pad, int d, const float* W, int64_t M, float* G,
                             float2* LP, cudaStream_t st, const int* guard) {
    if (M <= 0) return cudaSuccess;
    if (d_pad % 32 || d_pad < 32 || d_pad > kDenseMaxDim || M > (1LL << 30)) return cudaErrorInvalidValue;
    switch (d_pad / 32) {
#define LAPS_Q(n) \
    case n: return launch_q<n>(P, d, W, M, G, LP, st, guard);
        LAPS_Q(1) LAPS_Q(2) LAPS_Q(3) LAPS_Q(4) LAPS_Q(5) LAPS_Q(6) LAPS_Q(7) LAPS_Q(8)
        LAPS_Q(9) LAPS_Q(10) LAPS_Q(11) LAPS_Q(12) LAPS_Q(13) LAPS_Q(14) LAPS_Q(15) LAPS_Q(16)
#undef LAPS_Q
    }
    return cudaErrorInvalidValue;
}

}  // namespace laps
