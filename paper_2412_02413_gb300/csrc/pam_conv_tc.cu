// pam_conv_tc.cu -- tensor-core (tcgen05) 3x3 convolutions of the learned
// NCC-weight network, for rows of nx = 128 pixels. Forward: the first layer
// (5 -> 32, bias, ReLU), the hidden layers (32 -> 32, bias, ReLU) and the last
// layer (32 -> 1, bias, FP32 output). Input gradients: the same convolution of
// dY with the adjoint weights (1 -> 32 or 32 -> 32), zero where the layer's
// input activation, a ReLU output, is zero.
//
// One output row is a GEMM with M = 128 pixels, N = 32 output channels (16
// for the last layer, whose channels 1..15 carry zero weights) and K = 9 taps
// x the input channels (one chunk of 8 for the first layer, padded in shared
// memory with a zero chunk to the K step of 16):
//   y[j][o] = b[o] + sum_{u,v,c} x[i+u-1][j+v-1][c] w[o][c][u][v].
// Activations are stored chunked and padded, [C/8][nz+2][nx+2][8] BF16 per
// frame, so one padded input row of one chunk of 8 channels is 130 pixels x
// 16 bytes, contiguous. Copied as it is into shared memory, 8 consecutive
// pixels of it form one 8-row x 16-byte core matrix of the canonical K-major
// layout (no swizzle): the A operand of tap (u, v) for channel chunks (c, c+1)
// is the staged row i+u-1 starting at pixel v, i.e. a descriptor whose start
// address moves by 16 bytes per pixel, with SBO = 128 bytes (next 8 pixels)
// and LBO = 2080 bytes (next chunk of channels). No im2col is materialised.
// The B operand (weights) is resident: [tap][chunk][out channel][8] BF16.
// Each row accumulates 9 x (chunks / 2) MMAs (M = 128, K = 16) into one of two
// tensor-memory accumulator sets.
//
// One CTA per (16-row strip, frame), 6 warps:
//   warp 0: bulk copies of the strip's 18 input rows through a ring of 6 slots;
//   warp 1: the MMA chain of each output row (one elected lane issues);
//   warps 2-5 (2-9 with EXACT): the epilogue, each reading its quarter of the 128 TMEM lanes
//     (pixels), adding the bias, and storing BF16 after ReLU (or FP32 channel 0).
// All waits are bounded; on expiry the CTA sets the status word and drains.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pam_internal.h"
#include "pam_ptx.h"

namespace pam {
namespace {

using namespace ptx;

constexpr int W = 128, WP = W + 2;
constexpr int ROWS = 16;                       // output rows per CTA
constexpr int NSLOT = 6;                       // staged input rows
constexpr int CH_BYTES = WP * 16;              // one padded row of one chunk: 2080 B
// Epilogue warps: one per quarter of the pixels, or two when boundary cases are
// looked for (each then has half of the output channels).
constexpr int epi_warps(bool exact) { return exact ? 8 : 4; }
constexpr int threads(bool exact) { return 64 + 32 * epi_warps(exact); }
constexpr int QCAP = 64;                       // boundary cases an epilogue warp collects before it recomputes 32

// Shape of one layer: NCI input chunks in global memory, KCH staged chunks
// (at least 2: one K step), NCO GEMM columns.
template <int NCI, int NCO>
struct ConvShape {
    static constexpr int KCH = NCI < 2 ? 2 : NCI;
    static constexpr int ROW_BYTES = KCH * CH_BYTES;
    static constexpr int TAP_BYTES = KCH * NCO * 16;
    static constexpr int WT_BYTES = 9 * TAP_BYTES;
    static constexpr size_t SMEM = (size_t)WT_BYTES + (size_t)NSLOT * ROW_BYTES + 256 + 8 * QCAP * sizeof(unsigned short);
    // kind::f16, FP32 accumulate, A = B = BF16, both K-major, N = NCO, M = 128.
    static constexpr unsigned IDESC = ptx::umma_idesc(false, 128, NCO);
};

__device__ __forceinline__ unsigned pack2(float a, float b)
{
    unsigned r;
    asm("cvt.rn.bf16x2.f32 %0, %2, %1;\n" : "=r"(r) : "f"(a), "f"(b));
    return r;
}

// Two values to packed BF16 with the ReLU; a NaN gives +0, as fmaxf(v, 0) does.
__device__ __forceinline__ unsigned pack2_relu(float a, float b)
{
    unsigned r;
    asm("max.bf16x2 %0, %1, %2;\n" : "=r"(r) : "r"(pack2(a, b)), "r"(0u));
    return r;
}

// What the epilogue does with a row: bias and ReLU, bias and FP32 output, or
// the ReLU mask of an input gradient.
enum { TC_RELU = 0, TC_F32 = 1, TC_MASK = 2 };

// Each of two packed BF16 values where its mask (a ReLU output: zero or
// positive) is positive, else zero.
__device__ __forceinline__ unsigned masked2(unsigned v, unsigned m)
{
    const unsigned lo = (m & 0xFFFFu) != 0u && (m & 0x8000u) == 0u ? 0xFFFFu : 0u;
    const unsigned hi = (m >> 16) != 0u && (m & 0x80000000u) == 0u ? 0xFFFF0000u : 0u;
    return v & (lo | hi);
}

// One output in the CUDA-core kernels' order (pam_learn.cu, conv_cc_kernel): a
// chain of FP32 FMAs over the input channels and, within one, the nine taps.
// `in` points at the output's pixel in the first of its three padded input rows
// (chunk planes `plane` apart), `w` at the output channel's weights in the
// staged [tap][KCH][NCO][8].
template <int NCI, int KCH, int NCO>
__device__ float conv_chain(const uint4 *__restrict__ in, size_t plane, const uint8_t *w)
{
    float s = 0.0f;
#pragma unroll 1
    for (int c = 0; c < NCI; ++c) {
        uint4 x[9], q[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            x[t] = in[(size_t)c * plane + (size_t)(t / 3) * WP + t % 3];
            q[t] = *reinterpret_cast<const uint4 *>(w + (size_t)((t * KCH + c) * NCO) * 16);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const unsigned xw = k < 2 ? x[t].x : k < 4 ? x[t].y : k < 6 ? x[t].z : x[t].w;
                const unsigned qw = k < 2 ? q[t].x : k < 4 ? q[t].y : k < 6 ? q[t].z : q[t].w;
                s = fmaf(__uint_as_float((k & 1) ? xw & 0xFFFF0000u : xw << 16),
                         __uint_as_float((k & 1) ? qw & 0xFFFF0000u : qw << 16), s);
            }
    }
    return s;
}

// EXACT (training): the outputs are, but for rare cases, those of the CUDA-core
// kernel, so a gradient hardly depends on which of the two computed the
// activations. Both sum in FP32 and differ by the order only, which shows where a
// sum lies within that difference of a BF16 rounding boundary or of the ReLU's zero:
// those outputs (about one in a thousand) are recomputed by conv_chain. An
// epilogue warp collects them over its rows and recomputes 32 at a time, one
// per lane: recomputing each row's few at once left most lanes idle (32 -> 32
// layer, 16 frames of 512 x 128: 107 us forward and 185 us backward, against 59
// and 78 us, with packed checks 53 and 66; 36 us without EXACT).
// The window on either side is CHAIN_TOL times the largest final sum of the
// thread's 16 channels, and BIAS_TOL of the value itself for the rounding of the
// bias addition. It is not a bound. The two orders (a chain of up to 288 roundings,
// and the tensor core's 9 or 18 truncated steps) differ in proportion to the terms:
// by 1.5e-7 of the largest sum (one standard deviation, a sixth of the window) for
// trained and random weights, but by more of it where the terms cancel in all 16
// channels at once. An output may then be the tensor core's rounding: within the same
// n 2^-23 sum |x w| of the exact sum, n terms, before its rounding to BF16.
constexpr float CHAIN_TOL = 9.5367431640625e-7f;   // 2^-20
constexpr float BIAS_TOL = 2.384185791015625e-7f;  // 2^-22: two FP32 ulp at least

template <int NCI, int NCO, int EPI, bool EXACT>
__global__ void __launch_bounds__(threads(EXACT), EXACT ? 2 : 1)
conv_tc_kernel(const uint4 *__restrict__ in, const uint4 *__restrict__ wt, const float *__restrict__ bias,
               const uint4 *__restrict__ mask, void *__restrict__ out, int H, int *__restrict__ status)
{
    using CS = ConvShape<NCI, NCO>;
    constexpr int THREADS = threads(EXACT), EPW = epi_warps(EXACT), NO = 128 / EPW;   // output channels per epilogue thread
    constexpr int KCH = CS::KCH, ROW_BYTES = CS::ROW_BYTES, WT_BYTES = CS::WT_BYTES;
    extern __shared__ __align__(1024) uint8_t sm[];
    uint8_t *sW = sm;                                  // [9][KCH][NCO][8] BF16
    uint8_t *sRow = sm + WT_BYTES;                     // [NSLOT][KCH][130][8] BF16
    uint64_t *full = reinterpret_cast<uint64_t *>(sRow + NSLOT * ROW_BYTES);   // [NSLOT]
    uint64_t *sfree = full + NSLOT;                    // [NSLOT]
    uint64_t *afull = sfree + NSLOT;                   // [2]
    uint64_t *aempty = afull + 2;                      // [2]
    uint64_t *wbar = aempty + 2;                       // [1]
    uint64_t *dbar = wbar + 1;                         // [1] drain
    unsigned *tslot = reinterpret_cast<unsigned *>(dbar + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int strip = blockIdx.x, f = blockIdx.y;
    const int HP = H + 2;
    const int r_first = strip * ROWS;
    const int nr = min(ROWS, H - r_first);   // output rows of this CTA
    const int nin = nr + 2;                  // input rows (padded rows r_first .. r_first + nr + 1)

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                     "r"(64u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 32) {
        for (int s = 0; s < NSLOT; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&sfree[s], 1);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&afull[t], 1);
            mbar_init(&aempty[t], EPW);
        }
        mbar_init(wbar, 1);
        mbar_init(dbar, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if constexpr (NCI < KCH) {
        // staged chunks NCI..KCH-1 of every slot stay zero (the K padding);
        // make the generic-proxy stores visible to the tensor core
        for (int i = tid; i < NSLOT * (KCH - NCI) * CH_BYTES / 16; i += THREADS) {
            const int slot = i / ((KCH - NCI) * CH_BYTES / 16), r = i % ((KCH - NCI) * CH_BYTES / 16);
            reinterpret_cast<uint4 *>(sRow + slot * ROW_BYTES + NCI * CH_BYTES)[r] = make_uint4(0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *tslot;

    auto wait = [&](uint64_t *b, unsigned parity) -> bool {
        if (mbar_try_wait_sleep(b, parity)) return true;
        const long long t0 = clock64();
        while (!mbar_try_wait_sleep(b, parity)) {
            if (*abort_flag) return false;
            if (clock64() - t0 > (1ll << 31)) {
                *abort_flag = 1;
                atomicOr(status, 1);
                return false;
            }
        }
        return true;
    };

    if (warp == 0) {
        // ---------------- producer: weights, then the input rows ----------------
        int issued = 0;
        bool ok = true;
        if (lane == 0) {
            mbar_expect_tx(wbar, WT_BYTES);
            bulk_g2s(sW, wt, WT_BYTES, wbar);
            for (int k = 0; k < nin && ok; ++k) {
                const int s = k % NSLOT;
                if (k >= NSLOT) ok = wait(&sfree[s], (unsigned)(k / NSLOT - 1) & 1u);
                if (!ok) break;
                mbar_expect_tx(&full[s], NCI * CH_BYTES);
                const int prow = r_first + k;
                for (int c = 0; c < NCI; ++c)
                    bulk_g2s(sRow + s * ROW_BYTES + c * CH_BYTES, in + (((size_t)f * NCI + c) * HP + prow) * WP,
                              CH_BYTES, &full[s]);
                issued = k + 1;
            }
            if (!ok) {
                // let the copies in flight land before the CTA exits
                wait(wbar, 0);
                for (int k = issued - NSLOT < 0 ? 0 : issued - NSLOT; k < issued; ++k)
                    wait(&full[k % NSLOT], (unsigned)(k / NSLOT) & 1u);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ---------------- MMA issue ----------------
        bool ok = __all_sync(0xffffffffu, wait(wbar, 0));
        bool any = false;
        const unsigned wbase = smem_u32(sW), rbase = smem_u32(sRow);
        for (int r = 0; r < nr && ok; ++r) {
            // input rows r, r+1, r+2 (the first two were waited for by earlier rows)
            for (int k = (r == 0 ? 0 : r + 2); k <= r + 2 && ok; ++k)
                ok = __all_sync(0xffffffffu, wait(&full[k % NSLOT], (unsigned)(k / NSLOT) & 1u));
            const int t = r & 1;
            if (ok && r >= 2) ok = __all_sync(0xffffffffu, wait(&aempty[t], (unsigned)((r >> 1) - 1) & 1u));
            if (!ok) break;
            tc_fence_after();
            const unsigned d = tmem + (unsigned)(t * 32);
#pragma unroll
            for (int tap = 0; tap < 9; ++tap) {
                const int u = tap / 3, v = tap % 3;
                const unsigned arow = rbase + (unsigned)(((r + u) % NSLOT) * ROW_BYTES + v * 16);
#pragma unroll
                for (int h = 0; h < KCH / 2; ++h) {
                    const uint64_t a = umma_desc(arow + (unsigned)(2 * h * CH_BYTES), CH_BYTES, 128);
                    const uint64_t b = umma_desc(wbase + (unsigned)(tap * CS::TAP_BYTES + h * 2 * NCO * 16), NCO * 16, 128);
                    umma_elect(d, a, b, CS::IDESC, (tap | h) ? 1u : 0u);
                }
            }
            any = true;
            umma_commit_elect(&afull[t]);
            umma_commit_elect(&sfree[r % NSLOT]);
        }
        if (any) {   // this warp's MMAs end before the tensor memory is freed, whichever warp gave up
            umma_commit_elect(dbar);
            mbar_wait(dbar, 0);
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: TMEM -> bias + ReLU, or the mask -> BF16 ----------------
        const int quarter = warp & 3;
        const int j = 32 * quarter + lane;   // pixel = TMEM lane
        const int o0 = NO * ((warp - 2) >> 2);   // first output channel
        constexpr int NB = EPI == TC_F32 ? 1 : EPI == TC_RELU ? NO : 0;
        float b[NB ? NB : 1];
#pragma unroll
        for (int o = 0; o < NB; ++o) b[o] = bias[o0 + o];
        unsigned short *queue = reinterpret_cast<unsigned short *>(sRow + NSLOT * ROW_BYTES + 256) + (warp - 2) * QCAP;
        int n_queue = 0;   // entries: row of the strip << 12 | lane << 5 | output channel
        // Entries at .. at + n - 1 (n <= 32), one per lane; the warp has stored these outputs before.
        auto recompute = [&](int at0, int n) {
            if (lane < n) {
                const unsigned e = queue[at0 + lane];
                const int o = (int)(e & 31u), qj = 32 * quarter + (int)((e >> 5) & 31u), qr = r_first + (int)(e >> 12);
                float v = conv_chain<NCI, KCH, NCO>(in + ((size_t)f * NCI * HP + qr) * WP + qj, (size_t)HP * WP,
                                                    sW + (size_t)o * 16);
                if constexpr (EPI == TC_RELU) v = fmaxf(v + bias[o], 0.0f);
                reinterpret_cast<unsigned short *>(reinterpret_cast<uint4 *>(out) +
                                                   (((size_t)f * 4 + (o >> 3)) * HP + qr + 1) * WP + qj + 1)[o & 7] =
                    (unsigned short)(pack2(v, v) & 0xFFFFu);
            }
            __syncwarp();
        };
        for (int r = 0; r < nr; ++r) {
            const int t = r & 1;
            // the row's mask is read while its MMAs run
            const size_t at = (((size_t)f * 4 + o0 / 8) * HP + r_first + r + 1) * WP + (j + 1);
            uint4 mk[NO / 8];
            if constexpr (EPI == TC_MASK) {
#pragma unroll
                for (int ch = 0; ch < NO / 8; ++ch) mk[ch] = mask[at + (size_t)ch * HP * WP];
            }
            if (!__all_sync(0xffffffffu, wait(&afull[t], (unsigned)(r >> 1) & 1u))) break;
            tc_fence_after();
            const unsigned taddr = tmem + (unsigned)(t * 32) + ((unsigned)(32 * quarter) << 16);
            if constexpr (EPI == TC_F32) {
                unsigned a0;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n" : "=r"(a0) : "r"(taddr));
                asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&aempty[t]);
                reinterpret_cast<float *>(out)[((size_t)f * H + r_first + r) * W + j] = __uint_as_float(a0) + b[0];
            } else {
                float acc[NO];
#pragma unroll
                for (int o = 0; o < NO; o += 16) tmem_ld16(taddr + (unsigned)(o0 + o), acc + o);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&aempty[t]);
                uint4 *dst = reinterpret_cast<uint4 *>(out) + at;
                // w[i]: outputs 2 i and 2 i + 1 as packed BF16; d[i]: where the two ends of the window differ
                unsigned w[NO / 2], d[NO / 2], any = 0u;
                float tol = 0.0f;
                if constexpr (EXACT) {
#pragma unroll
                    for (int o = 0; o < NO; ++o) tol = fmaxf(tol, fabsf(acc[o]));
                    tol *= CHAIN_TOL;
                }
#pragma unroll
                for (int i = 0; i < NO / 2; ++i) {
                    float2 v = make_float2(acc[2 * i], acc[2 * i + 1]);
                    if constexpr (EPI == TC_RELU) v = __fadd2_rn(v, make_float2(b[2 * i], b[2 * i + 1]));
                    w[i] = EPI == TC_RELU ? pack2_relu(v.x, v.y) : pack2(v.x, v.y);
                    if constexpr (EXACT) {
                        // an activation is positive, so the two ends move apart; an input gradient has no bias
                        const float hi = EPI == TC_RELU ? 1.0f + BIAS_TOL : 1.0f, lo = EPI == TC_RELU ? 1.0f - BIAS_TOL : 1.0f;
                        const float2 up = __ffma2_rn(v, make_float2(hi, hi), make_float2(tol, tol));
                        const float2 dn = __ffma2_rn(v, make_float2(lo, lo), make_float2(-tol, -tol));
                        d[i] = EPI == TC_RELU ? pack2_relu(up.x, up.y) ^ pack2_relu(dn.x, dn.y)
                                              : pack2(up.x, up.y) ^ pack2(dn.x, dn.y);
                    }
                    if constexpr (EPI == TC_MASK) {   // masked outputs are zero either way
                        const uint4 q = mk[i >> 2];
                        const unsigned m = (i & 3) == 0 ? q.x : (i & 3) == 1 ? q.y : (i & 3) == 2 ? q.z : q.w;
                        w[i] = masked2(w[i], m);
                        if constexpr (EXACT) d[i] = masked2(d[i], m);
                    }
                    if constexpr (EXACT) any |= d[i];
                }
#pragma unroll
                for (int ch = 0; ch < NO / 8; ++ch)
                    dst[(size_t)ch * HP * WP] = make_uint4(w[4 * ch], w[4 * ch + 1], w[4 * ch + 2], w[4 * ch + 3]);
                unsigned redo = 0u;   // bit o: output o is too near a boundary
                if constexpr (EXACT) {
                    if (any != 0u) {
#pragma unroll
                        for (int i = 0; i < NO / 2; ++i) {
                            if (d[i] & 0xFFFFu) redo |= 1u << (2 * i);
                            if (d[i] >> 16) redo |= 1u << (2 * i + 1);
                        }
                    }
                }
                if constexpr (EXACT) {
                    while (true) {
                        const unsigned have = __ballot_sync(0xffffffffu, redo != 0u);
                        if (have == 0u) break;
                        if (redo != 0u) {
                            queue[n_queue + __popc(have & ((1u << lane) - 1u))] =
                                (unsigned short)(r << 12 | lane << 5 | (o0 + __ffs(redo) - 1));
                            redo &= redo - 1u;
                        }
                        n_queue += __popc(have);
                        __syncwarp();
                        if (n_queue >= 32) {
                            n_queue -= 32;
                            recompute(n_queue, 32);
                        }
                    }
                }
            }
        }
        if constexpr (EXACT) {
            __syncwarp();
            recompute(0, n_queue);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(64u) : "memory");
}

template <int NCI, int NCO, int EPI, bool EXACT>
cudaError_t set_tc_smem()
{
    return cudaFuncSetAttribute(conv_tc_kernel<NCI, NCO, EPI, EXACT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)ConvShape<NCI, NCO>::SMEM);
}

template <int NCI, int NCO, int EPI, bool EXACT>
cudaError_t launch_tc(const uint4 *in, const uint4 *wt, const float *bias, const uint4 *mask, void *out, int F, int H,
                      int *status, cudaStream_t st)
{
    dim3 grid((H + ROWS - 1) / ROWS, F);
    conv_tc_kernel<NCI, NCO, EPI, EXACT><<<grid, threads(EXACT), ConvShape<NCI, NCO>::SMEM, st>>>(in, wt, bias, mask, out, H,
                                                                                           status);
    return cudaGetLastError();
}

}  // namespace

cudaError_t prepare_conv_tc()
{
    cudaError_t e = set_tc_smem<1, 32, TC_RELU, false>();
    if (e == cudaSuccess) e = set_tc_smem<4, 32, TC_RELU, false>();
    if (e == cudaSuccess) e = set_tc_smem<4, 16, TC_F32, false>();
    if (e == cudaSuccess) e = set_tc_smem<1, 32, TC_RELU, true>();
    if (e == cudaSuccess) e = set_tc_smem<4, 32, TC_RELU, true>();
    if (e == cudaSuccess) e = set_tc_smem<1, 32, TC_MASK, true>();
    if (e == cudaSuccess) e = set_tc_smem<4, 32, TC_MASK, true>();
    return e;
}

cudaError_t launch_conv_tc(int layer, const uint4 *in, const uint4 *wt, const float *bias, void *out, int F, int H,
                           int *status, cudaStream_t st)
{
    if (layer == 0) return launch_tc<1, 32, TC_RELU, false>(in, wt, bias, nullptr, out, F, H, status, st);
    if (layer == 4) return launch_tc<4, 16, TC_F32, false>(in, wt, bias, nullptr, out, F, H, status, st);
    return launch_tc<4, 32, TC_RELU, false>(in, wt, bias, nullptr, out, F, H, status, st);
}

cudaError_t launch_conv_tc_exact(int layer, const uint4 *in, const uint4 *wt, const float *bias, uint4 *out, int F,
                                 int H, int *status, cudaStream_t st)
{
    if (layer == 0) return launch_tc<1, 32, TC_RELU, true>(in, wt, bias, nullptr, out, F, H, status, st);
    return launch_tc<4, 32, TC_RELU, true>(in, wt, bias, nullptr, out, F, H, status, st);
}

cudaError_t launch_conv_tc_grad(int layer, const uint4 *dY, const uint4 *wt, const uint4 *mask, uint4 *out, int F,
                                int H, int *status, cudaStream_t st)
{
    if (layer == 4) return launch_tc<1, 32, TC_MASK, true>(dY, wt, nullptr, mask, out, F, H, status, st);
    return launch_tc<4, 32, TC_MASK, true>(dY, wt, nullptr, mask, out, F, H, status, st);
}

}  // namespace pam
