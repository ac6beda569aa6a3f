// laps_logreg.cu -- FP32 SIMT gradient of the logistic-regression target for
// an ensemble of points (the all-FP32 form; also the adjusted phase of the
// mixed-precision form).  kp <= 128 runs the packed kernel, larger kp the plain one.
//
// Plain kernel: a block owns a tile of 64 chains and one range of data rows.  Its 64 x kp
// slice of W stays in shared memory; the data rows stream through shared
// memory 64 at a time.  Per chunk:
//   Z  = W_tile X_chunk^T      (64 x 64, thread tile 4 chains x 4 rows)
//   R  = y - sigmoid(Z), log p terms y z - softplus(z)   (registers)
//   G += R^T-tile X_chunk      (64 x kp, thread tile 4 chains x 4 NG coords)
// so Z and R live only in registers and a 17 KB shared tile.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "laps_device.cuh"
#include "laps_logreg.cuh"

namespace laps {

namespace {

constexpr int TM = 64;    // chains per block
constexpr int TN = 64;    // data rows per chunk
constexpr int NT = 256;   // threads
constexpr int RTS = TM + 4;  // row stride of the transposed R tile

template <int KP>
__global__ void __launch_bounds__(NT, KP <= 128 ? 2 : 1)
logreg_grad_f32_kernel(const float* __restrict__ W, int64_t M, const float* __restrict__ X,
                       const float* __restrict__ yv, int n, int rps, float inv_v,
                       float* __restrict__ gpart, float2* __restrict__ lpart, const int* __restrict__ guard) {
    if (guard != nullptr && *guard == 0) return;  // the iteration no longer runs
    constexpr int LD = KP + 4;   // padded row stride (floats) of the W and X tiles
    constexpr int NG = KP / 64;  // float4 column groups per thread in the G phase
    extern __shared__ __align__(16) float sm[];
    float* Ws = sm;                 // [TM][LD]
    float* Xs = Ws + TM * LD;       // [TN][LD]
    float* Rt = Xs + TN * LD;       // [TN][RTS]  R transposed: Rt[row][chain]
    float* wsq = Rt + TN * RTS;     // [TM] |w|^2

    const int tid = threadIdx.x;
    const int64_t m0 = (int64_t)blockIdx.x * TM;
    const int s = blockIdx.y;
    const int r_begin = s * rps;
    const int r_end = min(n, r_begin + rps);

    // W tile (rows beyond M are zero)
    for (int k = tid; k < TM * (KP / 4); k += NT) {
        const int r = k / (KP / 4), c4 = k - r * (KP / 4);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (m0 + r < M) v = *reinterpret_cast<const float4*>(W + (m0 + r) * KP + 4 * c4);
        *reinterpret_cast<float4*>(Ws + r * LD + 4 * c4) = v;
    }
    __syncthreads();
    if (s == 0) {  // |w|^2 for the prior term: 4 lanes per chain
        const int r = tid >> 2, q = tid & 3;
        float a = 0.0f;
        for (int k = q; k < KP; k += 4) a = fmaf(Ws[r * LD + k], Ws[r * LD + k], a);
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        if (q == 0) wsq[r] = a;
    }

    const int cr = tid >> 4;  // chains 4cr .. 4cr+3 of the tile
    const int dc = tid & 15;  // Z phase: rows dc + 16e;  G phase: columns 64q + 4dc .. +3
    float gacc[4][4 * NG];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int k = 0; k < 4 * NG; ++k) gacc[c][k] = 0.0f;
    ff lacc[4] = {ff_make(0.0f), ff_make(0.0f), ff_make(0.0f), ff_make(0.0f)};

    for (int row0 = r_begin; row0 < r_end; row0 += TN) {
        // ---- the chunk's data rows (rows past the range are zero and masked below)
        __syncthreads();
        for (int k = tid; k < TN * (KP / 4); k += NT) {
            const int r = k / (KP / 4), c4 = k - r * (KP / 4);
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (row0 + r < r_end) v = *reinterpret_cast<const float4*>(X + (size_t)(row0 + r) * KP + 4 * c4);
            *reinterpret_cast<float4*>(Xs + r * LD + 4 * c4) = v;
        }
        __syncthreads();
        // ---- Z = W X^T on the 4 x 4 thread tile
        float z[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) z[c][e] = 0.0f;
#pragma unroll 4
        for (int k = 0; k < KP; k += 4) {
            float4 wv[4], xv[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) wv[c] = *reinterpret_cast<const float4*>(Ws + (4 * cr + c) * LD + k);
#pragma unroll
            for (int e = 0; e < 4; ++e) xv[e] = *reinterpret_cast<const float4*>(Xs + (dc + 16 * e) * LD + k);
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    z[c][e] = fmaf(wv[c].x, xv[e].x, z[c][e]);
                    z[c][e] = fmaf(wv[c].y, xv[e].y, z[c][e]);
                    z[c][e] = fmaf(wv[c].z, xv[e].z, z[c][e]);
                    z[c][e] = fmaf(wv[c].w, xv[e].w, z[c][e]);
                }
        }
        // ---- epilogue: residuals and log-likelihood terms
        float lsum[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = row0 + dc + 16 * e;
            const bool ok = row < r_end;
            const float yn = ok ? yv[row] : 0.0f;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float zz = z[c][e];
                const float t = expf(-fabsf(zz));               // e^{-|z|} in (0, 1]
                const float sp = fmaxf(zz, 0.0f) + log1pf(t);   // softplus(z)
                const float inv = 1.0f / (1.0f + t);
                const float sig = zz >= 0.0f ? inv : t * inv;   // sigmoid(z)
                Rt[(dc + 16 * e) * RTS + 4 * cr + c] = ok ? yn - sig : 0.0f;
                lsum[c] += ok ? fmaf(yn, zz, -sp) : 0.0f;
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) lacc[c] = ff_add(lacc[c], lsum[c]);
        __syncthreads();
        // ---- G += R^T X over the chunk's rows
#pragma unroll 4
        for (int r = 0; r < TN; ++r) {
            const float4 rv = *reinterpret_cast<const float4*>(Rt + r * RTS + 4 * cr);
            const float rr[4] = {rv.x, rv.y, rv.z, rv.w};
#pragma unroll
            for (int q = 0; q < NG; ++q) {
                const float4 xv = *reinterpret_cast<const float4*>(Xs + r * LD + 64 * q + 4 * dc);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    gacc[c][4 * q + 0] = fmaf(rr[c], xv.x, gacc[c][4 * q + 0]);
                    gacc[c][4 * q + 1] = fmaf(rr[c], xv.y, gacc[c][4 * q + 1]);
                    gacc[c][4 * q + 2] = fmaf(rr[c], xv.z, gacc[c][4 * q + 2]);
                    gacc[c][4 * q + 3] = fmaf(rr[c], xv.w, gacc[c][4 * q + 3]);
                }
            }
        }
    }
    __syncthreads();  // wsq is visible (written before the loop; the loop may be empty)

    // ---- outputs: gradient partial (plus the prior on range 0) and log p partial
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const int64_t m = m0 + 4 * cr + c;
        // log p: the 16 threads of this chain group add their partials in a fixed order
        ff l = group_sum_ff<16>(lacc[c]);
        if (m >= M) continue;
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            const int col = 64 * q + 4 * dc;
            float4 v = make_float4(gacc[c][4 * q], gacc[c][4 * q + 1], gacc[c][4 * q + 2], gacc[c][4 * q + 3]);
            if (s == 0) {
                const float4 w = *reinterpret_cast<const float4*>(Ws + (4 * cr + c) * LD + col);
                v.x = fmaf(-w.x, inv_v, v.x);
                v.y = fmaf(-w.y, inv_v, v.y);
                v.z = fmaf(-w.z, inv_v, v.z);
                v.w = fmaf(-w.w, inv_v, v.w);
            }
            *reinterpret_cast<float4*>(gpart + ((size_t)s * M + m) * KP + col) = v;
        }
        if (dc == 0) {
            if (s == 0) l = ff_add(l, -0.5f * inv_v * wsq[4 * cr + c]);
            lpart[(size_t)s * M + m] = make_float2(l.hi, l.lo);
        }
    }
}

// ---------------------------------------------------------------- packed form
// The same contraction for kp <= 128 with packed binary32 pairs (fma.rn.f32x2),
// every sum in the plain kernel's order and every operation rounded as there, so that
// without ROUND the results are the plain kernel's bit for bit.  What bounds
// it is the FMA pipe: 2 M n d multiply-adds, of which the pipe retires 128 per clock
// and SM either way, but a packed instruction carries two, so half the issue slots
// are left for the operand loads and the epilogue.  A thread owns 8 chains x 4 rows
// of Z and 8 chains x 4 NG columns of G, so that an operand vector from shared
// memory feeds four to eight packed instructions:
//   Z: pairs of chains (c, c + 1), interleaved in the W tile; the data value is
//      duplicated into both halves; the loop stops at the last non-zero feature
//      (d rounded up to 4), not at the padded width;
//   G: pairs of columns, the residual stored twice by the epilogue.
// A target call (ROUND) rounds log p to binary32, so its log p need not be the plain
// kernel's sum bit for bit: Z pairs even and odd k (both operands come as pairs from
// 16-byte loads, no duplication) and the epilogue takes one log1p per four rows, of
// prod (1 + t) - 1 built up as e <- e + t + e t (no cancellation, so small t keep their
// relative precision; at most 15).
// 128 threads and 64 chains per block, two blocks per SM: one block's staging and
// epilogue overlap the other's contraction.
// Measured at d = 101, n = 10^4, M = 8192: gradient call 1083 -> 923 us in the plain
// kernel's order (kernel 1061 -> 911 us; FMA pipe 64% busy with 23% fewer multiply-adds
// in Z), 900 us with ROUND; the gradient's error against binary64 stays 2.3e-7 and
// log p's 2.8e-8 (relative norms).
constexpr int PT = 128;        // threads
constexpr int RTP = 2 * TM + 4;  // row stride of the duplicated R tile

template <int KP, bool ROUND>
__global__ void __launch_bounds__(PT, 2)
logreg_grad_f32p_kernel(const float* __restrict__ W, int64_t M, const float* __restrict__ X,
                        const float* __restrict__ yv, int n, int kz, int rps, float inv_v,
                        float* __restrict__ gpart, float2* __restrict__ lpart, const int* __restrict__ guard) {
    if (guard != nullptr && *guard == 0) return;  // the iteration no longer runs
    constexpr int LD = KP + 4;       // padded row stride (floats) of the X tile
    constexpr int LDW = 2 * KP + 4;  // and of the W tile's pairs of rows (not ROUND)
    constexpr int NG = KP / 64;      // float4 column groups per thread in the G phase
    extern __shared__ __align__(16) float sm[];
    float* Ws = sm;  // [TM / 2][LDW]  row cr + 8 i: chains (cr + 16 i, cr + 16 i + 8), pairs per k; ROUND: [TM][LD]
    float* Xs = Ws + (ROUND ? TM * LD : TM / 2 * LDW);  // [TN][LD]
    float* Rt = Xs + TN * LD;         // [TN][RTP]  Rt[row][32 i + 4 cr]: chain cr + 16 i twice, cr + 16 i + 8 twice
    float* wsq = Rt + TN * RTP;       // [TM] |w|^2
    ff* s_lp = reinterpret_cast<ff*>(wsq + TM);  // [8][2][32] log p of the upper half of the rows, a lane's chains

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t m0 = (int64_t)blockIdx.x * TM;
    const int s = blockIdx.y;
    const int r_begin = s * rps;
    const int r_end = min(n, r_begin + rps);
    // chain r of the tile at k: row (r & 7) + 8 (r >> 4), half (r >> 3) & 1
    auto wat = [&](int r, int k) -> float& {
        return ROUND ? Ws[r * LD + k] : Ws[((r & 7) + 8 * (r >> 4)) * LDW + 2 * k + ((r >> 3) & 1)];
    };

    // W tile (rows beyond M are zero)
    for (int k = tid; k < TM * (KP / 4); k += PT) {
        const int r = k / (KP / 4), c4 = k - r * (KP / 4);
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (m0 + r < M) v = *reinterpret_cast<const float4*>(W + (m0 + r) * KP + 4 * c4);
        wat(r, 4 * c4) = v.x;
        wat(r, 4 * c4 + 1) = v.y;
        wat(r, 4 * c4 + 2) = v.z;
        wat(r, 4 * c4 + 3) = v.w;
    }
    __syncthreads();
    if (s == 0)  // |w|^2 for the prior term: 4 lanes per chain
        for (int r = tid >> 2; r < TM; r += PT / 4) {
            const int q = tid & 3;
            float a = 0.0f;
            for (int k = q; k < KP; k += 4) a = fmaf(wat(r, k), wat(r, k), a);
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            if (q == 0) wsq[r] = a;
        }

    // a warp spans 4 chain groups x 8 rows (columns): its 16-byte operand loads touch
    // 4 or 8 distinct addresses in distinct banks
    const int cr = 4 * (warp & 1) + (lane >> 3);  // chains cr + 8 c
    const int dc = 8 * (warp >> 1) + (lane & 7);  // Z: rows dc + 16 e;  G: columns 64 q + 4 dc .. +3
    f32x2 gacc[8][2 * NG];
#pragma unroll
    for (int c = 0; c < 8; ++c)
#pragma unroll
        for (int k = 0; k < 2 * NG; ++k) gacc[c][k] = 0;
    ff lacc[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) lacc[c] = ff_make(0.0f);
    const float* wb = Ws + cr * (ROUND ? LD : LDW);
    const float* xb = Xs + dc * LD;

    for (int row0 = r_begin; row0 < r_end; row0 += TN) {
        // ---- the chunk's data rows (rows past the range are zero and masked below)
        __syncthreads();
        for (int k = tid; k < TN * (KP / 4); k += PT) {
            const int r = k / (KP / 4), c4 = k - r * (KP / 4);
            const uint32_t dst = (uint32_t)__cvta_generic_to_shared(Xs + r * LD + 4 * c4);
            const bool in = row0 + r < r_end;
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst),
                         "l"(X + (size_t)(in ? row0 + r : row0) * KP + 4 * c4), "r"(in ? 16 : 0)
                         : "memory");
        }
        float yn[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = row0 + dc + 16 * e;
            yn[e] = row < r_end ? yv[row] : 0.0f;
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // ---- Z = W X^T on the 8 x 4 thread tile, k in order (ROUND: even and odd k apart)
        f32x2 z[ROUND ? 8 : 4][4];
#pragma unroll
        for (int i = 0; i < (ROUND ? 8 : 4); ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) z[i][e] = 0;
        if constexpr (ROUND) {
#pragma unroll 2
            for (int k = 0; k < kz; k += 4) {
                ulonglong2 xv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) xv[e] = *reinterpret_cast<const ulonglong2*>(xb + 16 * e * LD + k);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const ulonglong2 wv = *reinterpret_cast<const ulonglong2*>(wb + 8 * c * LD + k);
#pragma unroll
                    for (int e = 0; e < 4; ++e) z[c][e] = fma2(wv.y, xv[e].y, fma2(wv.x, xv[e].x, z[c][e]));
                }
            }
        } else {
#pragma unroll 2
            for (int k = 0; k < kz; k += 4) {
                float4 xv[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) xv[e] = *reinterpret_cast<const float4*>(xb + 16 * e * LD + k);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    ulonglong2 wv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) wv[i] = *reinterpret_cast<const ulonglong2*>(wb + 8 * i * LDW + 2 * k + 4 * h);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float a = h == 0 ? xv[e].x : xv[e].z, b = h == 0 ? xv[e].y : xv[e].w;
                        const f32x2 aa = pack2(a, a), bb = pack2(b, b);
#pragma unroll
                        for (int i = 0; i < 4; ++i) z[i][e] = fma2(wv[i].y, bb, fma2(wv[i].x, aa, z[i][e]));
                    }
                }
            }
        }
        // ---- epilogue: residuals and log-likelihood terms
        auto epilogue = [&](auto full) {
            float lsum[8], lprod[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                lsum[c] = 0.0f;
                lprod[c] = 0.0f;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const bool ok = decltype(full)::value || row0 + dc + 16 * e < r_end;
                float4* dst = reinterpret_cast<float4*>(Rt + (dc + 16 * e) * RTP + 4 * cr);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float2 zp;
                    if constexpr (ROUND) {
                        const float2 za = unpack2(z[2 * i][e]), zb = unpack2(z[2 * i + 1][e]);
                        zp = make_float2(za.x + za.y, zb.x + zb.y);
                    } else {
                        zp = unpack2(z[i][e]);
                    }
                    float r[2];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float zz = h == 0 ? zp.x : zp.y;
                        const float t = expf(-fabsf(zz));               // e^{-|z|} in (0, 1]
                        const float inv = rcp_1_2(1.0f + t);
                        const float sig = zz >= 0.0f ? inv : t * inv;   // sigmoid(z)
                        r[h] = ok ? yn[e] - sig : 0.0f;
                        if constexpr (ROUND) {  // y z - max(z, 0); log(1 + t) below
                            lsum[2 * i + h] += ok ? fmaf(yn[e], zz, -fmaxf(zz, 0.0f)) : 0.0f;
                            const float e1 = lprod[2 * i + h], tk = ok ? t : 0.0f;
                            lprod[2 * i + h] = fmaf(e1, tk, tk) + e1;
                        } else {
                            const float sp = fmaxf(zz, 0.0f) + log1pf(t);  // softplus(z)
                            lsum[2 * i + h] += ok ? fmaf(yn[e], zz, -sp) : 0.0f;
                        }
                    }
                    dst[8 * i] = make_float4(r[0], r[0], r[1], r[1]);
                }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) lacc[c] = ff_add(lacc[c], ROUND ? lsum[c] - log1pf(lprod[c]) : lsum[c]);
        };
        if (row0 + TN <= r_end) epilogue(std::true_type{});
        else epilogue(std::false_type{});
        __syncthreads();
        // ---- G += R^T X over the chunk's rows, in order
#pragma unroll 2
        for (int r = 0; r < TN; ++r) {
            f32x2 rr[8];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(Rt + r * RTP + 32 * i + 4 * cr);
                rr[2 * i] = v.x;
                rr[2 * i + 1] = v.y;
            }
#pragma unroll
            for (int q = 0; q < NG; ++q) {
                const ulonglong2 xv = *reinterpret_cast<const ulonglong2*>(Xs + r * LD + 64 * q + 4 * dc);
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    gacc[c][2 * q] = fma2(rr[c], xv.x, gacc[c][2 * q]);
                    gacc[c][2 * q + 1] = fma2(rr[c], xv.y, gacc[c][2 * q + 1]);
                }
            }
        }
    }

    // ---- outputs: gradient partial (plus the prior on range 0) and log p partial.
    // log p: row dc + 8's partial (the warp two up, same lane) before the 8 lanes of a
    // chain, the order of the plain kernel's butterfly
    ff* s_w = s_lp + 32 * (warp & 1) + lane;
    if (warp >= 2)
#pragma unroll
        for (int c = 0; c < 8; ++c) s_w[64 * c] = lacc[c];
    __syncthreads();  // s_lp and wsq are visible (the loop may be empty)
    if (warp < 2)
#pragma unroll
        for (int c = 0; c < 8; ++c) lacc[c] = group_sum_ff<8>(ff_add(lacc[c], s_w[64 * c]));
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const int64_t m = m0 + cr + 8 * c;
        if (m >= M) continue;
#pragma unroll
        for (int q = 0; q < NG; ++q) {
            const int col = 64 * q + 4 * dc;
            const float2 v0 = unpack2(gacc[c][2 * q]), v1 = unpack2(gacc[c][2 * q + 1]);
            float4 v = make_float4(v0.x, v0.y, v1.x, v1.y);
            if (s == 0) {
                const float4 w = *reinterpret_cast<const float4*>(W + m * KP + col);
                v.x = fmaf(-w.x, inv_v, v.x);
                v.y = fmaf(-w.y, inv_v, v.y);
                v.z = fmaf(-w.z, inv_v, v.z);
                v.w = fmaf(-w.w, inv_v, v.w);
            }
            *reinterpret_cast<float4*>(gpart + ((size_t)s * M + m) * KP + col) = v;
        }
        if (warp < 2 && (lane & 7) == 0) {
            ff l = lacc[c];
            if (s == 0) l = ff_add(l, -0.5f * inv_v * wsq[cr + 8 * c]);
            lpart[(size_t)s * M + m] = make_float2(l.hi, l.lo);
        }
    }
}

// kp <= 128 has the packed kernel (its accumulators and Z tile need 250 registers at
// kp = 192 and above).  It takes the launch when some SM gets two blocks; below that an
// SM holds one block, whose four warps reach 83 of the FMA pipe's 128 lanes a clock, and the
// plain kernel's eight are faster (n = 262, d = 72, M = 198, 20 blocks: 15 steps of a run
// 787 against 847 us).  In the sampler both give the same bits, so the line between
// them is of speed alone; a target call (ROUND) adds in another order in the packed one.
template <int KP>
constexpr bool kPacked = KP <= 128;

template <int KP>
size_t f32_smem(bool packed) {
    const size_t tiles = (size_t)TM * (KP + 4) + (size_t)TN * (KP + 4) + TM;
    if (packed) return (tiles + (size_t)TN * RTP + 16 * TM) * sizeof(float);  // W: TM / 2 rows of 2 kp + 4
    return (tiles + (size_t)TN * RTS) * sizeof(float);
}

template <int KP>
cudaError_t launch_f32(const LogregData& D, const float* W, int64_t M, int S, bool round_lp, float* gpart,
                       float2* lpart, cudaStream_t st, const int* guard) {
    const int rps = (D.n + S - 1) / S;
    const dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)S);
    if constexpr (kPacked<KP>) {
        int dev = 0, nsm = 1;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if ((int64_t)grid.x * S > nsm) {
            const size_t smem = f32_smem<KP>(true);
            auto fn = round_lp ? logreg_grad_f32p_kernel<KP, true> : logreg_grad_f32p_kernel<KP, false>;
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
            fn<<<grid, PT, smem, st>>>(W, M, D.X, D.y, D.n, (D.d + 3) / 4 * 4, rps, D.inv_v, gpart, lpart, guard);
            return cudaGetLastError();
        }
    }
    const size_t smem = f32_smem<KP>(false);
    cudaError_t e = cudaFuncSetAttribute(logreg_grad_f32_kernel<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    logreg_grad_f32_kernel<KP><<<grid, NT, smem, st>>>(W, M, D.X, D.y, D.n, rps, D.inv_v, gpart, lpart, guard);
    return cudaGetLastError();
}

}  // namespace

namespace {
// blocks per SM the data split plans for: the plain kernel's (the packed one's is the same)
template <int KP>
int f32_blocks_per_sm() {
    int n = 0;
    if (cudaFuncSetAttribute(logreg_grad_f32_kernel<KP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)f32_smem<KP>(false)) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, logreg_grad_f32_kernel<KP>, NT, f32_smem<KP>(false)) !=
            cudaSuccess) {
        cudaGetLastError();
        n = 0;
    }
    return std::max(n, 1);
}
}  // namespace

int logreg_f32_splits(const LogregData& D, int64_t M, int nsm) {
    int bps = 1;
    switch (D.kp) {
    case 64: bps = f32_blocks_per_sm<64>(); break;
    case 128: bps = f32_blocks_per_sm<128>(); break;
    case 192: bps = f32_blocks_per_sm<192>(); break;
    case 256: bps = f32_blocks_per_sm<256>(); break;
    }
    const int64_t tiles = (M + TM - 1) / TM, slots = (int64_t)bps * std::max(nsm, 1);
    const int chunks = std::max(1, (D.n + TN - 1) / TN);
    // a block's time ~ its rows plus about one chunk of fixed work (the W tile in,
    // the partials out); the run's time ~ waves x that
    int best = 1;
    int64_t best_cost = -1;
    for (int S = 1; S <= std::min(16, chunks); ++S) {
        const int64_t waves = (tiles * S + slots - 1) / slots;
        const int64_t cost = waves * ((D.n + S - 1) / S + TN);
        if (best_cost < 0 || cost < best_cost) {
            best = S;
            best_cost = cost;
        }
    }
    return best;
}

cudaError_t logreg_grad_f32(const LogregData& D, const float* W, int64_t M, int S, bool round_lp, float* gpart,
                            float2* lpart, cudaStream_t st, const int* guard) {
    if (M <= 0) return cudaSuccess;
    if (S < 1 || S > 65535 || (M + TM - 1) / TM > 0x7fffffff) return cudaErrorInvalidValue;
    switch (D.kp) {
    case 64: return launch_f32<64>(D, W, M, S, round_lp, gpart, lpart, st, guard);
    case 128: return launch_f32<128>(D, W, M, S, round_lp, gpart, lpart, st, guard);
    case 192: return launch_f32<192>(D, W, M, S, round_lp, gpart, lpart, st, guard);
    case 256: return launch_f32<256>(D, W, M, S, round_lp, gpart, lpart, st, guard);
    }
    return cudaErrorInvalidValue;
}

}  // namespace laps
