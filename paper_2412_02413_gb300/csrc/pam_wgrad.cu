// pam_wgrad.cu -- weight gradients of the 3x3 convolutions of the learned
// NCC-weight network on the tensor cores (tcgen05, BF16 operands, FP32 sums).
//
// dW[o][c][u][v] = sum_{f,i,j} dY[f][o][i][j] X[f][c][i+u-1][j+v-1], db[o] = sum dY
// is, per output row i and column shift v, a GEMM whose K runs over the row's
// pixels: M = (row shift u, input channel c), N = output channel o. Activations
// and gradients are stored chunked and padded, BF16 [C/8][H+2][W+2][8], so a row
// of one chunk copied as it is into shared memory is a column of 8 x 8 core
// matrices of the MN-major layout without swizzle: 8 channels in 16 contiguous
// bytes, 16 bytes per pixel along K (LBO: the next 8 pixels, 128 bytes). The
// next 8 channels are the next chunk and, past a row's last chunk, the next
// staged row, at one stride (SBO): staged rows i, i+1, i+2 are the operand of the
// three row shifts at once, and a column shift moves the start address by 16
// bytes. Nothing is rearranged in memory.
//
// Work: one CTA per SM takes an equal contiguous share of the batch's rows
// (frame after frame). Warp 0 stages each input row (three output rows use it)
// and each dY row once, by bulk copies into two rings; warps 1-3 issue one column
// shift's W / 16 MMAs (M = 128, N = 32 or 16, K = 16) per output row each; warps 4-7
// add up db from the staged dY rows and, every SETK K steps, add the accumulators of
// the three column shifts to FP32 sums in registers, while the MMAs go on into a
// second set of accumulators. The hardware truncates the accumulators, a bias that
// grows with the chain: over 8 steps (4 in the last layer, whose terms are often of
// one sign and whose sums are one column to read) the error against 64-bit sums is
// that of FP32 FMAs or less at every width, over 32 steps the last layer's was 2 to 7
// times that (16 frames of 100 x 128, trained weights: 1.4e-7 of the gradient against
// 1.15e-6, and 1.5e-7 with FMAs). The CTA writes one partial; wgrad_reduce_kernel adds
// the CTAs' partials in order, so results do not depend on timing.
//
// A window of 16 groups of 8 channels is more than the three rows: the groups
// past them read whatever the following slots hold, which only reaches
// accumulator rows (or, with one dY chunk, columns) that nobody reads.
//
// Measured (GB300, 16 frames of 512 x 128): 49 us for 32 -> 32 channels, 45 us for
// the first layer and 50 us for the last (47, 43 and 43 with chains of 32 steps),
// where one issuing warp took 61 us, mma.sync 97 us (its rate) and the CUDA cores
// 689 us. Bound by the hand-offs and the issue of a row (0.8 us): a branch beside each
// MMA makes 61 us of it, while halving the MMAs, dropping the db sums, four
// accumulator sets or deeper rings change it by less than 5%, and DRAM runs at
// 3 TB/s. One MMA of N = 96 per 16 pixels, with dY staged once per column shift, took
// 61 us (three times the copies).
#include <cuda_runtime.h>
#include <stdint.h>

#include "pam_internal.h"
#include "pam_ptx.h"

namespace pam {
namespace {

using namespace ptx;

constexpr int NSX = 8, NSY = 6;    // ring slots of input rows and dY rows (NSY >= NSX - 2)
constexpr int THREADS = 256;
constexpr int GROUPS = 16;         // 8-channel groups of M = 128

// NCI input chunks, NCY dY chunks (of 8 channels).
template <int NCI, int NCY>
struct WG {
    static constexpr int NB = NCY == 1 ? 16 : 8 * NCY;     // GEMM columns (at least 16 for M = 128)
    static constexpr int VROWS = 3 * NCI * 8;              // accumulator rows in use
    static constexpr int SETK = NCY == 1 ? 4 : 8;          // K steps (of 16 pixels) of an accumulator
    static constexpr int HALVES = 8 / SETK;                // accumulators of a row of 128 pixels and column shift
    // input ring: NSX slots, the first two again behind the last (a window of
    // three rows is contiguous from any slot), and room for the rest of the window
    static constexpr int XSLOTS = NSX + 2;
    static constexpr int XCHUNKS = (NSX - 1) * NCI + GROUPS > XSLOTS * NCI ? (NSX - 1) * NCI + GROUPS : XSLOTS * NCI;
    static constexpr int YCHUNKS = NSY * NCY + 1;          // the second column group of NCY = 1 reads one further
    static_assert(HALVES == 1 || NB == 16, "one accumulator per column shift where all columns are read");
    static_assert(2 * 3 * HALVES * NB <= 256, "two accumulator sets in the tensor memory allocated");
    static constexpr size_t smem(int W) { return 1024 + (size_t)(XCHUNKS + YCHUNKS) * (W + 2) * 16; }
};

// kind::f16, FP32 accumulators, BF16 operands, both MN-major
constexpr unsigned idesc_mn(int n) { return umma_idesc(false, 128, n) | (1u << 15) | (1u << 16); }

// part: [gridDim.x][CO * CI * 9 + CO] partial sums in the parameter layout of
// the layer (w[o][c][3][3], then b[o]; CI, CO real channels).
template <int NCI, int NCY>
__global__ void __launch_bounds__(THREADS, 1)
wgrad_tc_kernel(const uint4 *__restrict__ X, const uint4 *__restrict__ dY, int F, int H, int W, int CI, int CO,
                float *__restrict__ part, int *__restrict__ status)
{
    using G = WG<NCI, NCY>;
    constexpr int NB = G::NB;
    extern __shared__ __align__(1024) uint8_t sm[];
    uint64_t *xfull = reinterpret_cast<uint64_t *>(sm);   // [NSX] input row has landed
    uint64_t *xfree = xfull + NSX;                        // [NSX] the MMAs (3 commits) that read it are done
    uint64_t *yfull = xfree + NSX, *yfree = yfull + NSY;  // [NSY] dY rows: 3 MMA warps and the 4 db warps
    uint64_t *afull = yfree + NSY, *aempty = afull + 2;   // [2] accumulator sets
    uint64_t *dbar = aempty + 2;                          // [3] drain
    unsigned *tslot = reinterpret_cast<unsigned *>(dbar + 3);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
    float *sdb = reinterpret_cast<float *>(sm + 512);     // [4 warps][32] db of each warp's pixels
    const unsigned CHB = (unsigned)(W + 2) * 16u;         // one row of one chunk
    uint8_t *sX = sm + 1024, *sY = sX + (size_t)G::XCHUNKS * CHB;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp == 0) tmem_alloc(tslot, 256u);
    if (tid == 32) {
        for (int s = 0; s < NSX; ++s) {
            mbar_init(&xfull[s], 1);
            mbar_init(&xfree[s], 3);
        }
        for (int s = 0; s < NSY; ++s) {
            mbar_init(&yfull[s], 1);
            mbar_init(&yfree[s], 7);
        }
        for (int t = 0; t < 2; ++t) {
            mbar_init(&afull[t], 3);
            mbar_init(&aempty[t], 4);
        }
        for (int v = 0; v < 3; ++v) mbar_init(&dbar[v], 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = *tslot;

    // Bounded wait that also gives up when another warp has.
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

    // An accumulator set: SETK K steps in each accumulator, of 2^lrps rows or of half a row.
    const int lrps = 16 * G::SETK > W ? 31 - __clz(16 * G::SETK / W) : 0;
    const int halves = W > 16 * G::SETK ? G::HALVES : 1;
    // Whether row `done` (of `rows`) of the share is the last of its set.
    auto last_of_set = [lrps](int done, int rows) { return ((done + 1) & ((1 << lrps) - 1)) == 0 || done + 1 == rows; };

    // The share's rows, in segments of one frame: n output rows from row a of
    // frame f use n + 2 staged input rows (counted by nx) and n dY rows (ny).
    const long long T = (long long)F * H;
    const long long r0 = T * blockIdx.x / gridDim.x, r1 = T * (blockIdx.x + 1) / gridDim.x;
    const int HP = H + 2, WP = W + 2;
    unsigned nx = 0, ny = 0;
    bool ok = true;

    if (warp == 0) {
        // ---------------- producer: lane c copies chunk c ----------------
        for (long long r = r0; r < r1 && ok;) {
            const int f = (int)(r / H), a = (int)(r - (long long)f * H);
            const int n = (int)min((long long)(H - a), r1 - r);
            for (int k = 0; k < n + 2; ++k) {
                const unsigned s = nx % NSX;
                const bool twice = s < 2;   // again behind the last slot
                if (nx >= NSX) ok = __all_sync(0xffffffffu, wait(&xfree[s], (nx / NSX - 1) & 1u));
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(&xfull[s], (twice ? 2u : 1u) * NCI * CHB);
                __syncwarp();
                if (lane < (twice ? 2 : 1) * NCI) {
                    const int c = lane % NCI;
                    bulk_g2s(sX + (size_t)((s + (lane >= NCI ? NSX : 0)) * NCI + c) * CHB,
                             X + (((size_t)f * NCI + c) * HP + a + k) * WP, CHB, &xfull[s]);
                }
                ++nx;
                if (k < 2) continue;
                const unsigned t = ny % NSY;   // dY row a + k - 2, padded row + 1
                if (ny >= NSY) ok = __all_sync(0xffffffffu, wait(&yfree[t], (ny / NSY - 1) & 1u));
                if (!ok) break;
                if (lane == 0) mbar_expect_tx(&yfull[t], NCY * CHB);
                __syncwarp();
                if (lane < NCY)
                    bulk_g2s(sY + (size_t)(t * NCY + lane) * CHB, dY + (((size_t)f * NCY + lane) * HP + a + k - 1) * WP,
                             CHB, &yfull[t]);
                ++ny;
            }
            r += n;
        }
        if (lane == 0) {
            if (*abort_flag) {   // the copies in flight land before the CTA exits
                for (unsigned k = nx < NSX ? 0 : nx - NSX; k < nx; ++k) mbar_wait(&xfull[k % NSX], (k / NSX) & 1u);
                for (unsigned k = ny < NSY ? 0 : ny - NSY; k < ny; ++k) mbar_wait(&yfull[k % NSY], (k / NSY) & 1u);
            }
        }
        __syncwarp();
    } else if (warp < 4) {
        // ---------------- MMA issue, column shift v ----------------
        const int v = warp - 1;
        const unsigned xb = smem_u32(sX), yb = smem_u32(sY);
        const int rows = (int)(r1 - r0);
        int done = 0;
        bool any = false;
        for (long long r = r0; r < r1 && ok;) {
            const int a = (int)(r % H);
            const int n = (int)min((long long)(H - a), r1 - r);
            for (int i = 0; i < n; ++i) {
                // input rows nx + i .. nx + i + 2 (the first two were waited for by earlier rows)
                for (unsigned k = i == 0 ? 0u : 2u; k < 3u && ok; ++k)
                    ok = wait(&xfull[(nx + i + k) % NSX], ((nx + i + k) / NSX) & 1u);
                const unsigned y = ny + (unsigned)i;
                if (ok) ok = wait(&yfull[y % NSY], (y / NSY) & 1u);
                const bool first = (done & ((1 << lrps) - 1)) == 0;
                const int set = done >> lrps, t = set & 1;
                if (ok && first && set >= 2) ok = wait(&aempty[t], (unsigned)((set >> 1) - 1) & 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                tc_fence_after();
                const unsigned arow = xb + ((nx + (unsigned)i) % NSX) * (NCI * CHB) + (unsigned)v * 16u;
                const unsigned brow = yb + (y % NSY) * (NCY * CHB) + 16u;   // dY has the border too
                const uint64_t da0 = umma_desc(arow, 128, CHB), db0 = umma_desc(brow, 128, CHB);
                // K step k of the row, `per` steps to an accumulator
                auto issue = [&](int k, int per) {
                    umma_elect(tmem + (unsigned)(((t * 3 + v) * G::HALVES + k / per) * NB), da0 + (uint64_t)(k * 16),
                               db0 + (uint64_t)(k * 16), idesc_mn(NB), (!first || k % per) ? 1u : 0u);
                };
                if (W == 128) {   // unrolled: issuing the MMAs is much of a row's time
#pragma unroll
                    for (int k = 0; k < 8; ++k) issue(k, G::SETK);
                } else {
#pragma unroll 4
                    for (int k = 0; k < W / 16; ++k) issue(k, 8);
                }
                any = true;
                if (last_of_set(done, rows)) umma_commit_elect(&afull[t]);
                umma_commit_elect(&xfree[(nx + i) % NSX]);
                if (i == n - 1) {   // the segment's last two rows are not used again
                    umma_commit_elect(&xfree[(nx + i + 1) % NSX]);
                    umma_commit_elect(&xfree[(nx + i + 2) % NSX]);
                }
                umma_commit_elect(&yfree[y % NSY]);
                ++done;
            }
            nx += (unsigned)n + 2u;
            ny += (unsigned)n;
            r += n;
        }
        if (any) {   // this warp's MMAs end before the tensor memory is freed, whichever warp gave up
            umma_commit_elect(&dbar[v]);
            mbar_wait(&dbar[v], 0);
        }
        __syncwarp();
    } else {
        // ---------------- sums ----------------
        const int quarter = warp & 3, ctid = tid - 128;
        float sum[3][NB == 16 ? 1 : NB];   // NCY = 1 has one real output channel
        constexpr int NO = NB == 16 ? 1 : NB;
#pragma unroll
        for (int v = 0; v < 3; ++v)
#pragma unroll
            for (int o = 0; o < NO; ++o) sum[v][o] = 0.0f;
        float db[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        // db: this thread's chunk and pixels (128 / NCY threads per chunk)
        const int ch = NCY == 1 ? 0 : ctid & (NCY - 1), p0 = ctid / NCY;
        const int rows = (int)(r1 - r0);
        for (int y = 0; y < rows; ++y) {
            if (!__all_sync(0xffffffffu, wait(&yfull[y % NSY], (unsigned)(y / NSY) & 1u))) break;
            const uint4 *row = reinterpret_cast<const uint4 *>(sY + (size_t)((y % NSY) * NCY + ch) * CHB) + 1;
            for (int p = p0; p < W; p += 128 / NCY) {
                const uint4 q = row[p];
                const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    db[2 * k] += __uint_as_float(w[k] << 16);
                    db[2 * k + 1] += __uint_as_float(w[k] & 0xFFFF0000u);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&yfree[y % NSY]);
            if (!last_of_set(y, rows)) continue;
            const int set = y >> lrps, t = set & 1;
            if (!__all_sync(0xffffffffu, wait(&afull[t], (unsigned)(set >> 1) & 1u))) break;
            tc_fence_after();
            const unsigned ta = tmem + (unsigned)(t * 3 * G::HALVES * NB) + ((unsigned)(32 * quarter) << 16);
            if constexpr (NB == 32) {
#pragma unroll
                for (int v = 0; v < 3; ++v) {
                    unsigned q[32];
                    tmem_ld32(ta + (unsigned)(v * NB), q);
                    tmem_wait_ld();
#pragma unroll
                    for (int o = 0; o < 32; ++o) sum[v][o] += __uint_as_float(q[o]);
                }
            } else {
                float q[3 * G::HALVES][4];
#pragma unroll
                for (int a = 0; a < 3 * G::HALVES; ++a) tmem_ld4(ta + (unsigned)(a * NB), q[a]);
                tmem_wait_ld();
#pragma unroll
                for (int a = 0; a < 3 * G::HALVES; ++a)
                    if (a % G::HALVES < halves) sum[a / G::HALVES][0] += q[a][0];
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&aempty[t]);
        }
        // accumulator row 8 NCI u + c: this thread's (u, c)
        float *dst = part + (size_t)blockIdx.x * ((size_t)CO * CI * 9 + CO);
        const int m = 32 * quarter + lane, u = m / (8 * NCI), c = m % (8 * NCI);
        if (!*abort_flag && m < G::VROWS && c < CI) {
#pragma unroll
            for (int v = 0; v < 3; ++v)
#pragma unroll
                for (int o = 0; o < NO; ++o)
                    if (o < CO) dst[((size_t)o * CI + c) * 9 + 3 * u + v] = sum[v][o];
        }
        // db: lanes of one chunk, then the four warps in order
#pragma unroll
        for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int d = 16; d >= NCY; d >>= 1) db[k] += __shfl_xor_sync(0xffffffffu, db[k], d);
        if (lane < NCY)
#pragma unroll
            for (int k = 0; k < 8; ++k) sdb[(warp - 4) * 32 + lane * 8 + k] = db[k];
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0) tmem_dealloc(tmem, 256u);
    if (!*abort_flag && tid < CO && tid < 32)
        part[(size_t)blockIdx.x * ((size_t)CO * CI * 9 + CO) + (size_t)CO * CI * 9 + tid] =
            ((sdb[tid] + sdb[32 + tid]) + sdb[64 + tid]) + sdb[96 + tid];
}

template <int NCI, int NCY>
cudaError_t launch_t(const uint4 *X, const uint4 *dY, int F, int H, int W, int CI, int CO, int ctas, float *part,
                     int *status, cudaStream_t st)
{
    static_assert(WG<NCI, NCY>::smem(128) <= 232448, "shared memory of the weight gradient");
    wgrad_tc_kernel<NCI, NCY><<<ctas, THREADS, WG<NCI, NCY>::smem(W), st>>>(X, dY, F, H, W, CI, CO, part, status);
    return cudaGetLastError();
}

template <int NCI, int NCY>
cudaError_t set_smem()
{
    return cudaFuncSetAttribute(wgrad_tc_kernel<NCI, NCY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)WG<NCI, NCY>::smem(128));
}

}  // namespace

cudaError_t prepare_wgrad()
{
    cudaError_t e = set_smem<1, 4>();
    if (e == cudaSuccess) e = set_smem<4, 4>();
    if (e == cudaSuccess) e = set_smem<4, 1>();
    return e;
}

int wgrad_ctas(int n_sms, int F, int H)
{
    // at least 4 output rows per CTA: a CTA stages 2 more input rows than it has output rows
    const long long n = ((long long)F * H + 3) / 4;
    return (int)(n < n_sms ? n : n_sms);
}

cudaError_t launch_wgrad(int layer, const uint4 *X, const uint4 *dY, int F, int H, int W, int ctas, float *part,
                         int *status, cudaStream_t st)
{
    if (layer == 0) return launch_t<1, 4>(X, dY, F, H, W, 5, 32, ctas, part, status, st);
    if (layer == 4) return launch_t<4, 1>(X, dY, F, H, W, 32, 1, ctas, part, status, st);
    return launch_t<4, 4>(X, dY, F, H, W, 32, 32, ctas, part, status, st);
}

}  // namespace pam
