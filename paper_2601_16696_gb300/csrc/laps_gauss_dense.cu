// laps_gauss_dense.cu -- log p and gradient of a Gaussian given by a dense
// precision matrix P (the rotated ill-conditioned Gaussian of the paper's
// Sec. 6):  log p = -1/2 x^T P x,  grad log p = -P x,  for the ensemble's
// points as one chains-by-coordinates contraction G = -W P.
//
// A block owns a few chains per warp (CW x warps, launch_q): their points stay in
// shared memory as pairs (x_k, x_k), P streams through shared memory kRows rows at a
// time (two buffers, cp.async), and lane l of the chain's warp accumulates the column
// pairs 2 l + 64 p in packed arithmetic (an odd multiple of 32 columns leaves one column
// a lane, in scalar arithmetic: a pair would idle half the warp).
//
// The target is ill-conditioned (condition number ~1e5 in the paper's
// experiment), so -P x cancels: a binary32 dot product loses ~1e-4 of max|g|.
// Each product therefore enters exactly into a float-float accumulator, two columns
// at a time (dense_add in laps_resident.cuh): the result is as accurate as a dot
// product in twice the working precision, rounded once.  log p sums x_o (P x)_o the
// same way, one warp butterfly per chain.
//
// What bounds it: ten FMA-pipe operations a product, and next to them the latency of the
// operand loads and of the sums' chains with one block of ten to sixteen warps an SM (M = 1500,
// d = 300: FMA pipe 58% busy, issue slots 40%).  Measured, us a launch, against scalar sums with
// a fixed sixteen chains a block (188 blocks on 152 SMs there): M = 1500, d = 300 88 -> 62;
// M = 4096, d = 200 79 -> 73; M = 4096, d = 100 24.5 -> 24.1.  The figures do not depend on the
// condition number.
#include <cuda_runtime.h>

#include <algorithm>

#include "laps_internal.h"

namespace laps {

namespace {
constexpr int kRows = 16;       // rows of P per chunk (d_pad is a multiple of 32)
constexpr int kMaxWarps = 16;

// W [M][dp] points (zero padded), P [dp][dp] symmetric (zero padded), dp = 32 Q.
// G [M][dp] receives -P x (zeros in the padding), LP [M] log p as float-float.
// nw: warps that hold chains (the block's other warps only stage).
template <int Q, int CW>
__global__ void __launch_bounds__(32 * kMaxWarps) gauss_dense_grad_kernel(const float* __restrict__ P, int d,
                                                                     const float* __restrict__ W, int64_t M, int nw,
                                                                     float* __restrict__ G,
                                                                     float2* __restrict__ LP,
                                                                     const int* __restrict__ guard) {
    if (guard != nullptr && *guard == 0) return;  // the iteration no longer runs
    constexpr int dp = 32 * Q, NP = Q / 2;  // pairs a lane; odd Q: one more column
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
    f32x2 hi[CW][NP + 1], lo[CW][NP + 1];
    float hi1[CW], lo1[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        hi1[c] = lo1[c] = 0.0f;
#pragma unroll
        for (int p = 0; p < NP; ++p) hi[c][p] = lo[c][p] = 0;
    }
    const f32x2 m1 = pack2(-1.0f, -1.0f);
    for (int k0 = 0, b = 0; k0 < d; k0 += kRows, b ^= 1) {
        if (k0 + kRows < d) {
            stage(k0 + kRows, b ^ 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        // rows past d of P are zero: they would add exact zeros, so stop at d (rounded up to 2)
        const int kn = work ? min(kRows, d - k0) : 0;
        const float *Pc = Ps + b * kRows * dp + 2 * lane, *P1 = Ps + b * kRows * dp + 64 * NP + lane;
#pragma unroll 2
        for (int kk = 0; kk < kn; kk += 2) {
            ulonglong2 xx[CW], nx[CW];
#pragma unroll
            for (int c = 0; c < CW; ++c) {
                xx[c] = *reinterpret_cast<const ulonglong2*>(Xs + (ch0 + c) * 2 * dp + 2 * (k0 + kk));
                nx[c] = make_ulonglong2(mul2(xx[c].x, m1), mul2(xx[c].y, m1));
            }
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const f32x2 p0 = *reinterpret_cast<const f32x2*>(Pc + kk * dp + 64 * p);
                const f32x2 p1 = *reinterpret_cast<const f32x2*>(Pc + (kk + 1) * dp + 64 * p);
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    dense_add(xx[c].x, nx[c].x, p0, m1, hi[c][p], lo[c][p]);
                    dense_add(xx[c].y, nx[c].y, p1, m1, hi[c][p], lo[c][p]);
                }
            }
            if constexpr (Q % 2 == 1) {
                const float p0 = P1[kk * dp], p1 = P1[(kk + 1) * dp];
#pragma unroll
                for (int c = 0; c < CW; ++c) {
                    dense_add(unpack2(xx[c].x).x, p0, hi1[c], lo1[c]);
                    dense_add(unpack2(xx[c].y).x, p1, hi1[c], lo1[c]);
                }
            }
        }
        __syncthreads();  // the buffer may be overwritten
    }
    if (!work) return;
    // -P x of each chain and its log p
#pragma unroll
    for (int c = 0; c < CW; ++c) {
        const int ch = ch0 + c;
        const float* xs = Xs + ch * 2 * dp;
        ff l = ff_make(0.0f);
        auto add_lp = [&](int o, float r) {
            const float pr = xs[2 * o] * r;
            l = ff_add(l, ff{pr, fmaf(xs[2 * o], r, -pr)});
        };
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const int o = 2 * lane + 64 * p;
            const float2 r = unpack2(add2(hi[c][p], lo[c][p]));
            add_lp(o, r.x);
            add_lp(o + 1, r.y);
            if (ch < nc)
                *reinterpret_cast<float2*>(G + (m0 + ch) * dp + o) = make_float2(o < d ? -r.x : 0.0f, o + 1 < d ? -r.y : 0.0f);
        }
        if constexpr (Q % 2 == 1) {
            const int o = 64 * NP + lane;
            const float r = hi1[c] + lo1[c];
            add_lp(o, r);
            if (ch < nc) G[(m0 + ch) * dp + o] = o < d ? -r : 0.0f;
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const ff w{__shfl_xor_sync(0xffffffffu, l.hi, off), __shfl_xor_sync(0xffffffffu, l.lo, off)};
            l = ff_add(l, w);
        }
        if (lane == 0 && ch < nc) LP[m0 + ch] = make_float2(-0.5f * l.hi, -0.5f * l.lo);
    }
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
