// laps_logreg_mma.cu -- the logistic-regression ensemble gradient on the
// 5th-generation tensor cores (tcgen05, BF16 operands, FP32 accumulation in
// tensor memory), for the unadjusted phase of the mixed-precision form.
//
// A CTA owns 128 chains (one MMA M tile) and one range of data rows, which it
// walks in chunks of 128 rows:
//   Z_c  = [W_hi | W_lo] [X_c | X_c]^T     128 x 128, K = 2 d   (TMEM, two buffers)
//   R_c  = y_c - sigmoid(Z_c)  (BF16, written into tensor memory by the epilogue)
//   G   += R_c X_c                          128 x d, K = 128     (TMEM; R read from TMEM)
// W = x is split into two BF16 terms (hi + lo carries ~16 significant bits),
// so the logits are those of the BF16-rounded data at nearly FP32 accuracy in
// x and log p stays smooth along a trajectory; R is a single BF16 term.
//
// Two epilogues.  The sampler's (FOLD = false) takes every row's logarithm and adds
// sixteen rows' terms in order, so that a run's log p does not depend on how rows are
// paired here; pairs of rows (j, j + 16) go through packed arithmetic side by side.  A
// target call on labels in {0, 1} (FOLD = true) rounds log p to binary32 anyway: it reads
// a copy of X whose label-1 rows are negated (exact), so that with z'' = (1 - 2 y) z the
// term is -softplus(z'') and the residual sigmoid(z''), loads no labels and takes one
// logarithm per sixteen rows, of the product of their 1 + t.
//
// What bounds it: the epilogue's special-function unit (ex2, reciprocal and, for the
// sampler, a logarithm per logit: 1/32 + 1/16 + 1/16 clocks and SM) and issue slots,
// next to the tensor pipe.  K and N stop at d rounded up to 16, not at the padded width;
// Z products of N = 128 run at the tensor peak, N = 64 ones at 63% of it; one copy of a
// data chunk serves both products (K-major for Z, MN-major for G).
// Measured at d = 101, n = 10^4, M = 8192 (kernel time): 105 us with 64-row chunks, two
// copies of a chunk, a scalar epilogue and one issuing thread; target call 76 us, sampler
// 86 us with the above; 60 and 81 us with an issuing warp per chain and two epilogue groups.
//
// Roles (640 threads): warp 0 loads W once and X chunks through a 4-stage ring
// with TMA (128-byte swizzle); warps 1 and 2 issue the Z and the G products; warps
// 4..19 are the epilogue, in two groups that take alternate chunks (one group's waits
// for Z and its tensor-memory loads overlap the other's arithmetic); warp w reads TMEM
// lanes 32 (w % 4) .. +31, i.e. chains, and half of the columns.  All waits are bounded: on expiry the CTA records
// ST_TIMEOUT in the status word, drains what it issued and frees its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "laps_device.cuh"
#include "laps_logreg.cuh"
#include "laps_rows.cuh"
#include "laps_tc.cuh"

namespace laps {

namespace {

constexpr int MT = 128;      // chains per CTA (MMA M)
constexpr int TNR = 128;     // data rows per chunk (MMA N of Z, K of G)
constexpr int NSTAGE = 4;    // X ring depth
constexpr int NTHR = 640;
constexpr int EPI_WARP0 = 4;  // first epilogue warp
constexpr int NEPI = 16;      // epilogue warps: 2 groups (even and odd chunks) x 2 column halves x 4 lane quarters

using namespace tc;

// SFU approximations in their flush-to-zero forms (the epilogue's arguments
// are never subnormal: 1 + t lies in [1, 2]; e^{-|z|} below 2^-126 flushes to 0)
__device__ __forceinline__ float ex2_ftz(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float lg2_ftz(float x) {
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_ftz(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&h);
}

struct MmaArgs {
    int64_t M;           // chains
    int n;               // data rows
    int rps;             // rows per split, a multiple of 64 (FOLD: of TNR)
    int d;               // features (padding columns of X and W are zero)
    float inv_v;         // 1 / prior variance
    const float* W32;    // [M][kp] FP32 x (for the prior terms)
    const float* yp;     // labels in pairs: 32 g + 2 j + {0, 1} holds rows 32 g + j and 32 g + 16 + j
    float* gpart;        // [S][M][kp]
    float2* lpart;       // [S][M]
    int* status;
    long long timeout_ns;
    const int* guard;    // nullable: 0 there means the iteration no longer runs
};

template <int KP>
struct Smem {
    static constexpr int NA = KP / 64;                    // 64-wide K atoms of one W term
    static constexpr uint32_t W_BYTES = 2u * NA * MT * 128;  // hi and lo
    static constexpr uint32_t ATOM = (uint32_t)TNR * 128;     // 64 features of one chunk
    static constexpr uint32_t STAGE = (uint32_t)NA * ATOM;
    static constexpr uint32_t OFF_W = 0;
    static constexpr uint32_t OFF_X = OFF_W + W_BYTES;
    static constexpr uint32_t OFF_BAR = OFF_X + NSTAGE * STAGE;
    static constexpr uint32_t OFF_LP = OFF_BAR + 256;      // [4][MT] float-float
    static constexpr uint32_t TOTAL = OFF_LP + 4 * MT * 8 + 1024;  // + alignment slack
    // tensor memory: Z buffers [0, 256), G [256, 256 + kp), R buffers (128 BF16 rows
    // per chain = 64 columns each) after G
    static constexpr uint32_t T_R = 2 * TNR + KP, TMEM_COLS = 512;
    static_assert(T_R + TNR <= TMEM_COLS, "tensor memory columns");
    static_assert(TOTAL <= 227 * 1024, "shared memory");
};

enum { B_WFULL = 0, B_XFULL = 1, B_XEMPTY = B_XFULL + NSTAGE, B_ZFULL = B_XEMPTY + NSTAGE,
       B_ZEMPTY = B_ZFULL + 2, B_RFULL = B_ZEMPTY + 2, B_REMPTY = B_RFULL + 2,
       B_GDONE = B_REMPTY + 2, B_DRAIN = B_GDONE + 1, NBAR = B_DRAIN + 2 };

template <int KP, bool FOLD>
__global__ void __launch_bounds__(NTHR, 1)
logreg_grad_mma_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                       const MmaArgs A) {
    if (A.guard != nullptr && *A.guard == 0) return;  // uniform: before any barrier or allocation
    using S = Smem<KP>;
    extern __shared__ __align__(1024) unsigned char mma_smem_raw[];
    __shared__ uint32_t s_tmem;
    __shared__ int s_fail;
    const uint32_t raw = smem_u32(mma_smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;  // 1024-byte aligned for the swizzle atoms
    unsigned char* gbase = mma_smem_raw + (base - raw);
    const uint32_t sW = base + S::OFF_W, sX = base + S::OFF_X;
    const uint32_t bars = base + S::OFF_BAR;
    ff* s_lp = reinterpret_cast<ff*>(gbase + S::OFF_LP);
    auto bar = [&](int k) { return bars + 8u * (uint32_t)k; };

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int64_t m0 = (int64_t)blockIdx.x * MT;
    const int split = blockIdx.y;
    const int r_begin = split * A.rps;
    const int r_end = min(A.n, r_begin + A.rps);
    const int nc = r_end > r_begin ? (r_end - r_begin + TNR - 1) / TNR : 0;
    const unsigned long long deadline = global_ns() + (unsigned long long)A.timeout_ns;

    if (tid == 32) {
        mbar_init(bar(B_WFULL), 1);
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(bar(B_XFULL + s), 1);
            mbar_init(bar(B_XEMPTY + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(B_ZFULL + b), 1);
            mbar_init(bar(B_ZEMPTY + b), NEPI / 2);
            mbar_init(bar(B_RFULL + b), NEPI / 2);
            mbar_init(bar(B_REMPTY + b), 1);
        }
        mbar_init(bar(B_GDONE), 1);
        mbar_init(bar(B_DRAIN), 1);
        mbar_init(bar(B_DRAIN + 1), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                     "r"(S::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
    const uint32_t tZ = tmem, tG = tmem + 2 * TNR, tR = tmem + S::T_R;

    if (warp == 0) {
      if (lane == 0) {
        // ------------------------------------------------ TMA producer
        bool ok = true;
        mbar_expect_tx(bar(B_WFULL), S::W_BYTES);
        for (int a = 0; a < 2 * S::NA; ++a)  // hi atoms then lo atoms: columns 64a of [hi | lo]
            tma_load_2d(sW + (uint32_t)a * (MT * 128), &tmW, 64 * a, (int)m0, bar(B_WFULL));
        int issued = 0;
        for (int c = 0; c < nc && ok; ++c) {
            const int st = c % NSTAGE;
            if (!mbar_wait(bar(B_XEMPTY + st), ((c / NSTAGE) & 1) ^ 1, deadline)) { ok = false; break; }
            const uint32_t dst = sX + (uint32_t)st * S::STAGE;
            mbar_expect_tx(bar(B_XFULL + st), S::STAGE);
            const int row = r_begin + c * TNR;
            for (int a = 0; a < S::NA; ++a)
                tma_load_2d(dst + (uint32_t)a * S::ATOM, &tmX, 64 * a, row, bar(B_XFULL + st));  // rows past n: 0
            issued = c + 1;
        }
        if (!ok) atomicExch(&s_fail, 1);
        // wait (bounded) for the copies this thread issued, whatever the other roles did: one of
        // them may have given up before it waited for the last chunks, and a CTA must not end
        // while copies into its shared memory are in flight
        const unsigned long long d2 = global_ns() + drain_ns(A.timeout_ns);
        mbar_wait(bar(B_WFULL), 0, d2);
        for (int c = max(0, issued - NSTAGE); c < issued; ++c)
            mbar_wait(bar(B_XFULL + c % NSTAGE), (c / NSTAGE) & 1, d2);
      }
      __syncwarp();
    } else if (warp <= 2) {
        // ------------------------------------------------ MMA issuers: warp 1 Z, warp 2 G
        // (the whole warp runs the loop, one elected lane issues).  A warp each, so that the
        // waits, fences and commits of one chain do not hold up the other's products: with one
        // thread for both, the tensor pipe stood idle for 40% of each chunk's 1344 clocks.
        const int k16 = (A.d + 15) / 16;  // K steps of one term of Z; N of G
        bool ok = true;
        if (warp == 1) {
            constexpr uint32_t ID_Z = idesc_bf16(MT, TNR);
            const uint64_t dX = sw128_desc(sX), dW = sw128_desc(sW);
            ok = mbar_wait_warp(bar(B_WFULL), 0, deadline);
            for (int c = 0; c < nc && ok; ++c) {
                const int st = c % NSTAGE, zb = c & 1;
                ok = mbar_wait_warp(bar(B_XFULL + st), (c / NSTAGE) & 1, deadline) &&
                     mbar_wait_warp(bar(B_ZEMPTY + zb), ((c >> 1) & 1) ^ 1, deadline);
                if (!ok) break;
                tc_fence_after();
                const uint64_t bX = dX + (uint64_t)((uint32_t)st * S::STAGE >> 4);
                const uint32_t dZ = tZ + (uint32_t)zb * TNR;
                if (elect_one()) {
#pragma unroll
                    for (int part = 0; part < 2; ++part)
#pragma unroll
                        for (int kk = 0; kk < KP / 16; ++kk)
                            if (kk < k16)
                                tc_mma(dZ, dW + (((uint32_t)(part * S::NA + kk / 4) * (MT * 128) + 32u * (kk % 4)) >> 4),
                                       bX + (((uint32_t)(kk / 4) * S::ATOM + 32u * (kk % 4)) >> 4), ID_Z,
                                       part + kk > 0 ? 1u : 0u);
                    tc_commit(bar(B_ZFULL + zb));
                }
                __syncwarp();
            }
        } else {
            const uint32_t ID_G = idesc_bf16(MT, 16 * k16, true);
            const uint64_t dXmn = sw128_mn_desc(sX, S::ATOM);
            for (int c = 0; c < nc && ok; ++c) {
                const int rb = c & 1, st = c % NSTAGE;
                ok = mbar_wait_warp(bar(B_XFULL + st), (c / NSTAGE) & 1, deadline) &&
                     mbar_wait_warp(bar(B_RFULL + rb), (c >> 1) & 1, deadline);
                if (!ok) break;
                tc_fence_after();
                const uint32_t aR = tR + (uint32_t)rb * (TNR / 2);
                const uint64_t bX = dXmn + (uint64_t)((uint32_t)st * S::STAGE >> 4);
                if (elect_one()) {
#pragma unroll
                    for (int kk = 0; kk < TNR / 16; ++kk)
                        tc_mma_ts(tG, aR + 8u * kk, bX + (2048u * kk >> 4), ID_G, (c > 0 || kk > 0) ? 1u : 0u);
                    tc_commit(bar(B_REMPTY + rb));
                    tc_commit(bar(B_XEMPTY + st));
                    if (c == nc - 1) tc_commit(bar(B_GDONE));
                }
                __syncwarp();
            }
            if (nc == 0 && elect_one()) mbar_arrive(bar(B_GDONE));
        }
        if (!ok) {
            if (elect_one()) {
                atomicExch(&s_fail, 1);
                tc_commit(bar(B_DRAIN + warp - 1));  // everything this warp issued has completed once it arrives
                mbar_wait(bar(B_DRAIN + warp - 1), 0, global_ns() + drain_ns(A.timeout_ns));
            }
            __syncwarp();
        }
    } else if (warp >= EPI_WARP0 && warp < EPI_WARP0 + NEPI) {
        // ------------------------------------------------ epilogue
        const int q = warp & 3;                 // TMEM lane quarter: chains 32q .. 32q+31
        constexpr int ZC = 32;                  // Z columns of one pass (two passes a warp)
        const int h = (warp - EPI_WARP0) >> 2;
        const int grp = h >> 1, half = h & 1;   // chunks c = grp (mod 2); Z columns 64 half .. + 63
        const int rt = 32 * q + lane;           // this thread's chain in the tile
        const uint32_t lane_off = (uint32_t)(32 * q) << 16;
        const f32x2 one2 = pack2(1.0f, 1.0f), m1 = pack2(-1.0f, -1.0f);
        const f32x2 nln2 = pack2(-0.6931471805599453f, -0.6931471805599453f);
        ff lp = ff_make(0.0f);
        bool ok = true;
        for (int c = grp; c < nc && ok; c += 2) {
            const int zb = grp, rb = grp;  // Z and R buffers of this group
            if (!mbar_wait_warp(bar(B_ZFULL + zb), (c >> 1) & 1, deadline)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int pass = 0; pass < 2; ++pass) {
            const int col0 = 64 * half + ZC * pass;
            const int row0 = r_begin + c * TNR + col0;
            const int nlive = min(ZC, max(0, r_end - row0));
            float z[ZC];
            tmem_ld32(tZ + lane_off + (uint32_t)(zb * TNR + col0), z);
            if (pass == 1) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(B_ZEMPTY + zb));
            }
            // Fast SFU approximations (this form serves the unadjusted phase only):
            // t = e^{-|z|}, sigmoid = (z >= 0 ? 1 : t) / (1 + t), softplus = max(z, 0) +
            // log(1 + t)
            uint32_t pr[ZC / 2];
            if constexpr (FOLD) {
                // Rows past n have z = 0 exactly: their sigmoid meets a zero data row, their
                // log 2 is taken off below.  The pairs' halves accumulate apart.
                f32x2 prod = one2, msum = 0;
#pragma unroll
                for (int j = 0; j < ZC; j += 2) {
                    const float t0 = ex2_ftz(-1.4426950408889634f * fabsf(z[j]));
                    const float t1 = ex2_ftz(-1.4426950408889634f * fabsf(z[j + 1]));
                    const f32x2 opt = add2(pack2(t0, t1), one2);
                    const float2 o = unpack2(opt);
                    const float2 r = unpack2(mul2(pack2(z[j] >= 0.0f ? 1.0f : t0, z[j + 1] >= 0.0f ? 1.0f : t1),
                                                  pack2(rcp_ftz(o.x), rcp_ftz(o.y))));
                    prod = mul2(prod, opt);
                    msum = add2(msum, pack2(fmaxf(z[j], 0.0f), fmaxf(z[j + 1], 0.0f)));
                    pr[j / 2] = pack_bf16(-r.x, -r.y);
                }
                const float2 ps = unpack2(prod), ms = unpack2(msum);
                const float l0 = fmaf(0.6931471805599453f, lg2_ftz(ps.x) - (float)((ZC - nlive) / 2), ms.x);
                const float l1 = fmaf(0.6931471805599453f, lg2_ftz(ps.y) - (float)((ZC - nlive + 1) / 2), ms.y);
                lp = ff_add(ff_add(lp, -l0), -l1);
            } else {
                f32x2 lsum = 0;  // rows row0 .. + 15 and row0 + 16 .. + 31, each in order
                const ulonglong2* yp = reinterpret_cast<const ulonglong2*>(A.yp + row0);
                auto body = [&](auto full) {
#pragma unroll
                    for (int j = 0; j < ZC / 2; j += 2) {
                        f32x2 yy[2] = {0, 0}, rr[2];
                        if (decltype(full)::value || nlive > j) {
                            const ulonglong2 v = __ldg(yp + j / 2);
                            yy[0] = v.x;
                            yy[1] = v.y;
                        }
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const float z0 = z[j + e], z1 = z[j + e + ZC / 2];
                            const float t0 = ex2_ftz(-1.4426950408889634f * fabsf(z0));
                            const float t1 = ex2_ftz(-1.4426950408889634f * fabsf(z1));
                            const float2 o = unpack2(add2(pack2(t0, t1), one2));
                            const f32x2 sig = mul2(pack2(z0 >= 0.0f ? 1.0f : t0, z1 >= 0.0f ? 1.0f : t1),
                                                   pack2(rcp_ftz(o.x), rcp_ftz(o.y)));
                            const f32x2 nsp = fma2(pack2(lg2_ftz(o.x), lg2_ftz(o.y)), nln2,
                                                   pack2(fminf(-z0, 0.0f), fminf(-z1, 0.0f)));  // -softplus
                            f32x2 term = fma2(yy[e], pack2(z0, z1), nsp);
                            rr[e] = fma2(sig, m1, yy[e]);  // y - sigmoid
                            if (!decltype(full)::value) {  // rows past the range add nothing
                                const float2 tv = unpack2(term), rv = unpack2(rr[e]);
                                const bool a = j + e < nlive, b = j + e + ZC / 2 < nlive;
                                term = pack2(a ? tv.x : 0.0f, b ? tv.y : 0.0f);
                                rr[e] = pack2(a ? rv.x : 0.0f, b ? rv.y : 0.0f);
                            }
                            lsum = add2(lsum, term);
                        }
                        const float2 r0 = unpack2(rr[0]), r1 = unpack2(rr[1]);
                        pr[j / 2] = pack_bf16(r0.x, r1.x);
                        pr[j / 2 + ZC / 4] = pack_bf16(r0.y, r1.y);
                    }
                };
                if (nlive == ZC) body(std::true_type{});
                else body(std::false_type{});
                const float2 ls = unpack2(lsum);
                lp = ff_add(ff_add(lp, ls.x), ls.y);
            }
            if (pass == 0 && !mbar_wait_warp(bar(B_REMPTY + rb), ((c >> 1) & 1) ^ 1, deadline)) { ok = false; break; }
            // R row rt, data rows col0 .. col0 + 31 of the chunk: columns col0 / 2 .. of this lane's R buffer
            tmem_st16(tR + lane_off + (uint32_t)(rb * (TNR / 2) + col0 / 2), pr);
            }
            if (!ok) break;
            tmem_st_wait();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(B_RFULL + rb));
        }
        ok = ok && mbar_wait_warp(bar(B_GDONE), 0, deadline);
        const int64_t m = m0 + rt;
        const float* wrow = A.W32 + (size_t)(m < A.M ? m : 0) * KP;
        if (!ok) atomicExch(&s_fail, 1);
        if (ok) {
            tc_fence_after();
            // G columns [h kp/4, (h+1) kp/4) of chain m, plus the prior on split 0
            float* gout = A.gpart + ((size_t)split * A.M + (m < A.M ? m : 0)) * KP;
#pragma unroll
            for (int piece = 0; piece < KP / 64; ++piece) {
                float g[16];
                const int col = h * (KP / 4) + 16 * piece;
                tmem_ld16(tG + lane_off + (uint32_t)col, g);
                if (nc == 0 || col >= A.d)  // no chunk, or past the products' N (d rounded up to 16)
#pragma unroll
                    for (int k = 0; k < 16; ++k) g[k] = 0.0f;  // G was never written
                if (m < A.M) {
#pragma unroll
                    for (int j4 = 0; j4 < 4; ++j4) {
                        float4 v = make_float4(g[4 * j4], g[4 * j4 + 1], g[4 * j4 + 2], g[4 * j4 + 3]);
                        if (split == 0) {
                            const float4 w = *reinterpret_cast<const float4*>(wrow + col + 4 * j4);
                            v.x = fmaf(-w.x, A.inv_v, v.x);
                            v.y = fmaf(-w.y, A.inv_v, v.y);
                            v.z = fmaf(-w.z, A.inv_v, v.z);
                            v.w = fmaf(-w.w, A.inv_v, v.w);
                        }
                        *reinterpret_cast<float4*>(gout + col + 4 * j4) = v;
                    }
                }
            }
            // log p: the four column quarters of a chain meet in shared memory
            s_lp[h * MT + rt] = lp;
        }
        asm volatile("bar.sync 1, %0;" ::"r"(NEPI * 32) : "memory");  // every epilogue warp
        if (ok) {
            if (h == 0 && m < A.M) {
                ff l = s_lp[rt];
#pragma unroll
                for (int k = 1; k < 4; ++k) l = ff_add(l, s_lp[k * MT + rt]);
                if (split == 0) {
                    float w2 = 0.0f;
                    for (int k = 0; k < KP; k += 4) {
                        const float4 w = *reinterpret_cast<const float4*>(wrow + k);
                        w2 = fmaf(w.x, w.x, fmaf(w.y, w.y, fmaf(w.z, w.z, fmaf(w.w, w.w, w2))));
                    }
                    l = ff_add(l, -0.5f * A.inv_v * w2);
                }
                A.lpart[(size_t)split * A.M + m] = make_float2(l.hi, l.lo);
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (s_fail && tid == 0) atomicExch(A.status, ST_TIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(S::TMEM_COLS)
                     : "memory");
    }
}

// ------------------------------------------------------------------ host
// X in BF16 and, in Xf, the same with the rows of label 1 negated
__global__ void to_bf16_kernel(const float* __restrict__ X, const float* __restrict__ y, __nv_bfloat16* __restrict__ Xb,
                               __nv_bfloat16* __restrict__ Xf, int n, int kp) {
    const int64_t tot = (int64_t)n * kp;
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < tot;
         k += (int64_t)gridDim.x * blockDim.x) {
        const __nv_bfloat16 v = __float2bfloat16_rn(X[k]);
        Xb[k] = v;
        Xf[k] = y[k / kp] == 1.0f ? __hneg(v) : v;
    }
}
// the labels in pairs (rows past n: 0); *other = 1 if some label is neither 0 nor 1
__global__ void pair_labels_kernel(const float* __restrict__ y, int n, int n32, float* __restrict__ yp,
                                   int* __restrict__ other) {
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n32; k += gridDim.x * blockDim.x) {
        const float v = k < n ? y[k] : 0.0f;
        yp[(k & ~31) + 2 * (k & 15) + ((k >> 4) & 1)] = v;
        if (!(v == 0.0f || v == 1.0f)) *other = 1;
    }
}

// caller's points [M][d] -> the FP32 [M][kp] copy and the BF16 hi | lo [M_pad][2 kp] copy
__global__ void pack_points_kernel(const float* __restrict__ x, RowIndex r, int d, float* __restrict__ W32,
                                   __nv_bfloat16* __restrict__ Wb) {
    for_elements(
        r, [&](int64_t m, int i) { return i < d ? x[m * d + i] : 0.0f; },
        [&](float v, int64_t k, int64_t m, int i) {
            W32[k] = v;
            const __nv_bfloat16 hi = __float2bfloat16_rn(v);
            Wb[m * 2 * r.w + i] = hi;
            Wb[m * 2 * r.w + r.w + i] = __float2bfloat16_rn(v - __bfloat162float(hi));
        });
}

template <int KP, bool FOLD>
cudaError_t launch_mma(const CUtensorMap& mw, const CUtensorMap& mx, const MmaArgs& a, dim3 grid, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(logreg_grad_mma_kernel<KP, FOLD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Smem<KP>::TOTAL);
    if (e != cudaSuccess) return e;
    logreg_grad_mma_kernel<KP, FOLD><<<grid, NTHR, Smem<KP>::TOTAL, st>>>(mw, mx, a);
    return cudaGetLastError();
}

}  // namespace

cudaError_t logreg_pack_points(const float* x, int64_t M, int d, int kp, float* W32, void* Wb,
                               cudaStream_t st) {
    const RowIndex r = row_index(M, kp);
    pack_points_kernel<<<row_blocks(r), 256, 0, st>>>(x, r, d, W32, reinterpret_cast<__nv_bfloat16*>(Wb));
    return cudaGetLastError();
}

bool logreg_mma_supported(int kp) { return kp == 64 || kp == 128; }

size_t logreg_mma_smem(int kp) { return kp == 64 ? Smem<64>::TOTAL : Smem<128>::TOTAL; }

cudaError_t logreg_mma_prepare(LogregData& D) {
    if (!logreg_mma_supported(D.kp)) return cudaErrorInvalidValue;
    EncodeTiled enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    // one allocation: Xb, Xf, the paired labels, the flag of other labels
    const size_t nb = (size_t)D.n * D.kp * sizeof(__nv_bfloat16);
    const int n32 = (D.n + 31) / 32 * 32;
    cudaError_t e = cudaMalloc(&D.Xb, 2 * nb + (size_t)n32 * sizeof(float) + sizeof(int));
    if (e != cudaSuccess) return e;
    D.Xf = static_cast<char*>(D.Xb) + nb;
    D.yp = reinterpret_cast<float*>(static_cast<char*>(D.Xb) + 2 * nb);
    int* other = reinterpret_cast<int*>(D.yp + n32);
    int h_other = 0;
    e = cudaMemset(other, 0, sizeof(int));
    if (e == cudaSuccess) {
        pair_labels_kernel<<<std::min(1024, (n32 + 255) / 256), 256>>>(D.y, D.n, n32, D.yp, other);
        to_bf16_kernel<<<std::min(4096, (int)((D.n * (int64_t)D.kp + 255) / 256)), 256>>>(
            D.X, D.y, reinterpret_cast<__nv_bfloat16*>(D.Xb), reinterpret_cast<__nv_bfloat16*>(D.Xf), D.n, D.kp);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h_other, other, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return e;
    D.bin = h_other == 0;
    // [n][kp], boxes of 64 features x 128 rows (rows past n read as zero)
    if (!encode_bf16_2d(D.tmX, D.Xb, (uint64_t)D.kp, (uint64_t)D.n, 64, TNR) ||
        !encode_bf16_2d(D.tmXf, D.Xf, (uint64_t)D.kp, (uint64_t)D.n, 64, TNR))
        return cudaErrorInvalidValue;
    return cudaSuccess;  // the copy of the flag waited for both kernels
}

cudaError_t logreg_mma_wmap(void* tmW, const void* Wb, int64_t M_pad, int kp) {
    EncodeTiled enc = encoder();
    if (!enc) return cudaErrorNotSupported;
    const cuuint32_t es[2] = {1, 1};
    const cuuint64_t dims[2] = {(cuuint64_t)(2 * kp), (cuuint64_t)M_pad};
    const cuuint64_t strides[1] = {(cuuint64_t)(2 * kp) * 2};
    const cuuint32_t box[2] = {64, MT};
    if (enc(reinterpret_cast<CUtensorMap*>(tmW), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(Wb), dims,
            strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

int logreg_mma_splits(const LogregData& D, int64_t M, int nsm, bool fold, int* rps_out) {
    const int64_t tiles = (M + MT - 1) / MT;
    const int unit = fold ? TNR : 64;
    int S = (int)std::max<int64_t>(1, nsm / std::max<int64_t>(1, tiles));
    const int chunks = (D.n + unit - 1) / unit;
    S = std::max(1, std::min(S, chunks));
    int rps = ((D.n + S - 1) / S + unit - 1) / unit * unit;
    S = (D.n + rps - 1) / rps;
    if (rps_out) *rps_out = rps;
    return S;
}

cudaError_t logreg_grad_mma(const LogregData& D, const void* tmW, const float* W32, int64_t M, int S,
                            int rps, bool fold, float* gpart, float2* lpart, int* status, long long timeout_ns,
                            cudaStream_t st, const int* guard) {
    if (M <= 0) return cudaSuccess;
    MmaArgs a;
    a.M = M;
    a.n = D.n;
    a.d = D.d;
    a.rps = rps;
    a.inv_v = D.inv_v;
    a.W32 = W32;
    a.yp = D.yp;
    a.gpart = gpart;
    a.lpart = lpart;
    a.status = status;
    a.timeout_ns = timeout_ns;
    a.guard = guard;
    const dim3 grid((unsigned)((M + MT - 1) / MT), (unsigned)S);
    const CUtensorMap& mw = *reinterpret_cast<const CUtensorMap*>(tmW);
    const CUtensorMap& mx = *reinterpret_cast<const CUtensorMap*>(fold ? D.tmXf : D.tmX);
    if (D.kp == 64) return fold ? launch_mma<64, true>(mw, mx, a, grid, st) : launch_mma<64, false>(mw, mx, a, grid, st);
    if (D.kp == 128)
        return fold ? launch_mma<128, true>(mw, mx, a, grid, st) : launch_mma<128, false>(mw, mx, a, grid, st);
    return cudaErrorInvalidValue;
}

}  // namespace laps
