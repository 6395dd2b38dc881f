// pam_wgrad.cu -- weight gradients of the 3x3 convolutions of the learned
// NCC-weight network on the tensor cores (mma.sync, BF16 operands, FP32 sums).
//
// dW[o][c][u][v] = sum_{f,i,j} dY[f][o][i][j] X[f][c][i+u-1][j+v-1], db[o] = sum dY
// is, per output row, a GEMM whose K runs over the row's pixels: M = (tap,
// input channel), N = output channel. Activations and gradients are stored
// chunked and padded, BF16 [C/8][H+2][W+2][8], so the 8 channels of one chunk
// at 8 consecutive pixels are an 8 x 8 matrix of 16-byte rows that
// ldmatrix.trans reads as (channel, pixel) fragments; a tap's column shift
// only moves the row addresses by 16 bytes per pixel and its row shift picks
// another staged row, so nothing is rearranged in memory.
//
// Why mma.sync and not tcgen05: N is 32 (8 for the last layer), and a tcgen05
// MMA of M = 128, N = 32 reads its 4 KB A tile from shared memory in 32 clocks
// for 16 clocks of tensor work, so both reach about the same rate here, near
// the time the two tensors take from HBM, and this form serves every width.
//
// Work: one CTA per SM takes an equal contiguous share of the batch's rows
// (frame after frame); thread 0 stages each input row (three output rows use
// it) and each dY row once through two rings of bulk copies, so that 12 warps
// keep up to 168 registers each (a 13th, a producer of its own, would leave
// 128 and spill). The warps are GROUPS x SPLITS: a group owns a part of the (tap, chunk) tiles, a
// split every SPLITS-th group of 16 pixels of the row. At the end the splits
// are added in order and the CTA writes one partial; wgrad_reduce_kernel adds the
// CTAs' partials in order, so results do not depend on timing.
//
// Measured (GB300, 16 frames of 512 x 128): 97 us for 32 -> 32 channels, 56
// and 55 us for the first and last layers, against 689, 197 and 86 us on the
// CUDA cores; bound by the mma.sync rate.
#include <cuda_runtime.h>
#include <stdint.h>

#include "pam_internal.h"
#include "pam_ptx.h"

namespace pam {
namespace {

using namespace ptx;

constexpr int NSX = 8, NSY = 6;   // ring slots of input rows and dY rows (NSY >= NSX - 2)

// NCI input chunks, NCY dY chunks (of 8 channels). TILES m16 tiles of two
// (tap, chunk) blocks each.
template <int NCI, int NCY>
struct WG {
    static constexpr int BLOCKS = 9 * NCI;
    static constexpr int TILES = (BLOCKS + 1) / 2;
    static constexpr int GROUPS = TILES * NCY > 40 ? 3 : 1;   // accumulators per thread: 4 TILES NCY / GROUPS
    static constexpr int SPLITS = GROUPS == 3 ? 4 : 8;
    static constexpr int TPG = TILES / GROUPS;
    static_assert(TPG * GROUPS == TILES, "tiles divide among the groups");
    static constexpr int WARPS = GROUPS * SPLITS;
    static constexpr int THREADS = 32 * WARPS;
    static constexpr int NR = (TPG + 1) * NCY * 4;     // floats per thread of the split reduction (tiles, db)
    static constexpr size_t ring(int W) { return (size_t)(NSX * NCI + NSY * NCY) * (W + 2) * 16; }
    static constexpr size_t red() { return (size_t)GROUPS * NR * 32 * 4; }
    static constexpr size_t smem(int W) { return 256 + (ring(W) > red() ? ring(W) : red()); }
};

__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm2t(unsigned (&r)[2], unsigned addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};\n"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// part: [gridDim.x][CO * CI * 9 + CO] partial sums in the parameter layout of
// the layer (w[o][c][3][3], then b[o]; CI, CO real channels).
template <int NCI, int NCY>
__global__ void __launch_bounds__(WG<NCI, NCY>::THREADS, 1)
wgrad_tc_kernel(const uint4 *__restrict__ X, const uint4 *__restrict__ dY, int F, int H, int W, int CI, int CO,
                float *__restrict__ part, int *__restrict__ status)
{
    using G = WG<NCI, NCY>;
    constexpr int TPG = G::TPG;
    extern __shared__ __align__(128) uint8_t sm[];
    uint64_t *xfull = reinterpret_cast<uint64_t *>(sm);   // [NSX] input row has landed
    uint64_t *xfree = xfull + NSX;                        // [NSX] every warp is done with it
    uint64_t *yfull = xfree + NSX, *yfree = yfull + NSY;  // [NSY] the same for dY rows
    const unsigned CHB = (unsigned)(W + 2) * 16u;         // one row of one chunk
    uint8_t *sX = sm + 256, *sY = sX + (size_t)NSX * NCI * CHB;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        for (int s = 0; s < NSX; ++s) {
            mbar_init(&xfull[s], 1);
            mbar_init(&xfree[s], G::WARPS);
        }
        for (int s = 0; s < NSY; ++s) {
            mbar_init(&yfull[s], 1);
            mbar_init(&yfree[s], G::WARPS);
        }
        mbar_fence_init();
    }
    __syncthreads();

    const long long T = (long long)F * H;
    const long long r0 = T * blockIdx.x / gridDim.x, r1 = T * (blockIdx.x + 1) / gridDim.x;
    const int HP = H + 2, WP = W + 2;
    bool ok = true;

    // Producer (thread 0): the rows of each segment (one frame's part of the
    // share) in order; input row k of a segment comes with the dY row of output
    // row k - 2. `seen` is the first input row that the thread's own warp still
    // needs: at most NSX - 1 rows from there are staged, so the slot to fill held
    // a row that the other warps finished two of their rows ago.
    unsigned px = 0, py = 0;      // rows issued
    long long pr = r0;            // next segment's first row
    int pf = 0, pa = 0, pn = 0, pk = 0;
    auto issue = [&](unsigned seen) {
        while (ok && px < seen + NSX - 1) {
            if (pk == (pn ? pn + 2 : 0)) {   // next segment
                if (pr >= r1) return;
                pf = (int)(pr / H);
                pa = (int)(pr - (long long)pf * H);
                pn = (int)min((long long)(H - pa), r1 - pr);
                pr += pn;
                pk = 0;
            }
            const unsigned s = px % NSX;
            if (px >= NSX) ok = mbar_wait(&xfree[s], (px / NSX - 1) & 1u);
            if (!ok) return;
            mbar_expect_tx(&xfull[s], NCI * CHB);
            for (int c = 0; c < NCI; ++c)
                bulk_g2s(sX + (size_t)(s * NCI + c) * CHB, X + (((size_t)pf * NCI + c) * HP + pa + pk) * WP, CHB,
                         &xfull[s]);
            ++px;
            if (++pk < 3) continue;
            const unsigned t = py % NSY;         // dY row pa + pk - 3, padded row + 1
            if (py >= NSY) ok = mbar_wait(&yfree[t], (py / NSY - 1) & 1u);
            if (!ok) return;
            mbar_expect_tx(&yfull[t], NCY * CHB);
            for (int c = 0; c < NCY; ++c)
                bulk_g2s(sY + (size_t)(t * NCY + c) * CHB, dY + (((size_t)pf * NCY + c) * HP + pa + pk - 2) * WP, CHB,
                         &yfull[t]);
            ++py;
        }
    };

    const int grp = warp / G::SPLITS, split = warp % G::SPLITS;
    const bool with_db = grp == 0;
    float acc[TPG + 1][NCY][4];   // the last tile's rows are all sum_k dY (a tile of ones), for db
#pragma unroll
    for (int t = 0; t <= TPG; ++t)
#pragma unroll
        for (int n = 0; n < NCY; ++n)
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[t][n][k] = 0.0f;

    {
        // Row of the lane's 8 x 8 matrix in an ldmatrix.x4: matrices are (block 0,
        // pixels 0-7), (block 1, 0-7), (block 0, 8-15), (block 1, 8-15) for A and
        // (chunk n, 0-7), (n, 8-15), (n + 1, 0-7), (n + 1, 8-15) for B.
        const int mi = lane >> 3;
        const unsigned a_px = (unsigned)((lane & 7) + 8 * (mi >> 1)), b_px = (unsigned)((lane & 7) + 8 * (mi & 1));
        // byte offset of the lane's block inside the three staged rows: row shift u
        // (a slot index, resolved per row), and chunk and column shift
        int a_u[TPG];
        unsigned a_off[TPG];
#pragma unroll
        for (int t = 0; t < TPG; ++t) {
            int blk = 2 * (grp * TPG + t) + (mi & 1);
            if (blk >= G::BLOCKS) blk = G::BLOCKS - 1;   // odd count: the spare rows are dropped at the end
            const int tap = blk / NCI, c = blk % NCI;
            a_u[t] = tap / 3;
            a_off[t] = (unsigned)c * CHB + ((unsigned)(tap % 3) + a_px) * 16u;
        }
        const unsigned b_off = (NCY > 1 ? (unsigned)(mi >> 1) * CHB : 0u) + (1u + b_px) * 16u;   // dY has the border too
        const unsigned ones[4] = {0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u};
        const unsigned xb = smem_u32(sX), yb = smem_u32(sY);
        unsigned nx = 0, ny = 0;   // rows of earlier segments
        for (long long r = r0; r < r1 && ok;) {
            const int a = (int)(r % H);
            const int n = (int)min((long long)(H - a), r1 - r);
            for (int i = 0; i < n && ok; ++i) {
                if (tid == 0) issue(nx + (unsigned)i);
                // input rows nx + i .. nx + i + 2 (the first two were waited for by earlier rows)
                for (int k = i == 0 ? 0 : 2; k < 3 && ok; ++k)
                    ok = mbar_wait(&xfull[(nx + i + k) % NSX], ((nx + i + k) / NSX) & 1u);
                const unsigned y = ny + (unsigned)i;
                if (ok) ok = mbar_wait(&yfull[y % NSY], (y / NSY) & 1u);
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                unsigned xrow[3];
#pragma unroll
                for (int u = 0; u < 3; ++u) xrow[u] = xb + ((nx + (unsigned)(i + u)) % NSX) * (NCI * CHB);
                const unsigned yrow = yb + (y % NSY) * (NCY * CHB) + b_off;
                for (int ks = split; ks < W / 16; ks += G::SPLITS) {
                    unsigned b[NCY][2];
                    if constexpr (NCY > 1) {
#pragma unroll
                        for (int q = 0; q < NCY; q += 2) {
                            unsigned v[4];
                            ldsm4t(v, yrow + (unsigned)q * CHB + (unsigned)ks * 256u);
                            b[q][0] = v[0]; b[q][1] = v[1]; b[q + 1][0] = v[2]; b[q + 1][1] = v[3];
                        }
                    } else {
                        ldsm2t(b[0], yrow + (unsigned)ks * 256u);
                    }
#pragma unroll
                    for (int t = 0; t < TPG; ++t) {
                        unsigned av[4];
                        const unsigned row = a_u[t] == 0 ? xrow[0] : a_u[t] == 1 ? xrow[1] : xrow[2];
                        ldsm4t(av, row + a_off[t] + (unsigned)ks * 256u);
#pragma unroll
                        for (int q = 0; q < NCY; ++q) mma16816(acc[t][q], av, b[q][0], b[q][1]);
                    }
                    if (with_db) {
#pragma unroll
                        for (int q = 0; q < NCY; ++q) mma16816(acc[TPG][q], ones, b[q][0], b[q][1]);
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&xfree[(nx + i) % NSX]);
                    if (i == n - 1) {   // the segment's last two rows are not used again
                        mbar_arrive(&xfree[(nx + i + 1) % NSX]);
                        mbar_arrive(&xfree[(nx + i + 2) % NSX]);
                    }
                    mbar_arrive(&yfree[y % NSY]);
                }
            }
            nx += (unsigned)n + 2u;
            ny += (unsigned)n;
            r += n;
        }
        if (!ok && lane == 0) atomicOr(status, 1);
    }
    if (__syncthreads_or(!ok)) {
        if (tid == 0) {   // the copies in flight land before the CTA exits
            for (unsigned k = px < NSX ? 0 : px - NSX; k < px; ++k) mbar_wait(&xfull[k % NSX], (k / NSX) & 1u);
            for (unsigned k = py < NSY ? 0 : py - NSY; k < py; ++k) mbar_wait(&yfull[k % NSY], (k / NSY) & 1u);
        }
        return;
    }
    // every row has been read: the rings' memory is free

    // the splits' sums added to split 0's, in order
    float *red = reinterpret_cast<float *>(sX) + (size_t)grp * (G::NR * 32);
    for (int s = 1; s < G::SPLITS; ++s) {
        if (split == s) {
#pragma unroll
            for (int t = 0; t <= TPG; ++t)
#pragma unroll
                for (int q = 0; q < NCY; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) red[((t * NCY + q) * 4 + k) * 32 + lane] = acc[t][q][k];
        }
        __syncthreads();
        if (split == 0) {
#pragma unroll
            for (int t = 0; t <= TPG; ++t)
#pragma unroll
                for (int q = 0; q < NCY; ++q)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[t][q][k] += red[((t * NCY + q) * 4 + k) * 32 + lane];
        }
        __syncthreads();
    }
    if (split != 0) return;
    // fragment (k): block row lane / 4 (+ 8 for k >= 2: the tile's second block), column 2 (lane % 4) + (k & 1)
    float *dst = part + (size_t)blockIdx.x * ((size_t)CO * CI * 9 + CO);
    const int row = lane >> 2, col = 2 * (lane & 3);
#pragma unroll
    for (int t = 0; t < TPG; ++t)
#pragma unroll
        for (int q = 0; q < NCY; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int blk = 2 * (grp * TPG + t) + (k >> 1);
                const int tap = blk / NCI, c = (blk % NCI) * 8 + row, o = q * 8 + col + (k & 1);
                if (blk < G::BLOCKS && c < CI && o < CO) dst[((size_t)o * CI + c) * 9 + tap] = acc[t][q][k];
            }
    if (with_db && row == 0) {
#pragma unroll
        for (int q = 0; q < NCY; ++q)
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int o = q * 8 + col + k;
                if (o < CO) dst[(size_t)CO * CI * 9 + o] = acc[TPG][q][k];
            }
    }
}

template <int NCI, int NCY>
cudaError_t launch_t(const uint4 *X, const uint4 *dY, int F, int H, int W, int CI, int CO, int ctas, float *part,
                     int *status, cudaStream_t st)
{
    using G = WG<NCI, NCY>;
    wgrad_tc_kernel<NCI, NCY><<<ctas, G::THREADS, G::smem(W), st>>>(X, dY, F, H, W, CI, CO, part, status);
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
