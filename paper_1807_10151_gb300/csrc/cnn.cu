// Learned perturbation network (not part of the paper: a small CNN that
// proposes the TV-nonascending direction of the superiorization step).
//
// Network: five 3x3 convolutions (zero padding), channels
//   16 (x / rms(x), tbar scaled to unit RMS, fourteen zeros) -> 32 -> 32 -> 32 -> 32 -> 1,
// ReLU after the first four; the output is added to the scaled tbar input
// (a residual around the plain direction).  Activations are BF16 in planes of
// eight channels (below), weights BF16, accumulation FP32.
//
// Every convolution (forward, and the input-gradient pass of training, which
// is a convolution with the flipped, transposed kernel) is an implicit GEMM on
// the 5th-generation tensor cores: a CTA walks down a strip of 128 columns with
// the input rows in a shared-memory ring and the packed weights (N = Cout,
// K = 9 * Cin) beside them, one thread issues one tcgen05.mma per tap and 16
// channels (M = 128 pixels), each reading the staged rows through a descriptor
// shifted by the tap's column offset (no im2col copy), into an FP32
// tensor-memory accumulator, and four warps read their 32 lanes back with
// tcgen05.ld for the epilogue (bias, ReLU or ReLU-mask, BF16 store).  The
// weight gradient is a contraction over pixels on the same tensor cores (both
// operands MN-major from the staged rows), accumulated per CTA in tensor
// memory and summed over CTAs in a fixed order.  Adam keeps FP32 master weights.
//
// Layout of an activation tensor of 8 c channels: [image][row -1 .. ny][plane of
// 8 channels][column][8], columns pitched at act_pitch(nx) with 8 columns of
// zeros on the left, the columns nx .. round_up(nx, 16) - 1 and the rows -1 and ny
// zero as well (written once, at creation).  One plane of one staged row, 130
// columns from j0 - 1 on, is then one contiguous run of 2080 bytes, so a row
// arrives by c bulk copies with the zero padding in place, and the epilogue's
// stores (16 bytes per lane, lanes on consecutive columns) are whole lines.  In
// the NHWC layout this replaced, a plane of a row was a TMA box of 130 separate
// 16-byte pieces, loaded three times (once per output row it touches): that, not
// the tensor cores, set the time (a 32 -> 32 layer of 8 x 512^2 took 122 us, 45 us
// now; the whole inference 657 against 309 us).
#include <math.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "tc.cuh"

namespace supcg {

constexpr int kCnnLayers = 5;
constexpr int kCh = 32;     // hidden channels
constexpr int kInCh = 16;   // stored input channels (2 used; 16 so that one tap fills one K = 16 step)
constexpr int kTile = 128;  // pixels per MMA tile


// layer l (0-based): storage channels of its input, real input channels, output channels
__host__ __device__ constexpr int l_cin(int l) { return l == 0 ? kInCh : kCh; }
__host__ __device__ constexpr int l_cin_real(int l) { return l == 0 ? 2 : kCh; }
__host__ __device__ constexpr int l_cout(int l) { return l == kCnnLayers - 1 ? 1 : kCh; }
__host__ __device__ constexpr int l_nout(int l) { return l == kCnnLayers - 1 ? 16 : kCh; }   // MMA N

enum { EPI_RELU = 0, EPI_LAST = 1, EPI_MASK = 2 };

__host__ __device__ constexpr int act_pitch(int nx) { return 8 + (nx + 15) / 16 * 16; }   // columns per plane row
// Index of the first column (8 elements per column) of a plane row; i from -1 to ny.
__host__ __device__ __forceinline__ size_t act_row(long long img, int i, int c8, int ch8, int ny, int pitch)
{
    return (((size_t)img * (ny + 2) + (i + 1)) * ch8 + c8) * (size_t)pitch + 8;
}

struct ConvArgs {
    const __nv_bfloat16 *in;    // CIN channels
    const __nv_bfloat16 *w;     // [3 NOUT][3 CIN] packed in core-matrix order (k_pack_weights)
    const float *bias;          // [>= NOUT] (RELU, LAST)
    __nv_bfloat16 *out_bf;      // 32 channels (RELU, MASK)
    float *out_f;               // one channel, [count][ny][nx] (LAST)
    const float *resid;         // [count][ny][nx], scaled by rscale[3 img + 1] and added to output channel 0 (LAST)
    const float *rscale;
    const __nv_bfloat16 *mask;  // 32 channels: keep where mask > 0 (MASK)
    int ny, nx, count;
    int tiles, segs, seg_rows;  // strips of 128 columns per image row, runs of rows per strip, rows per run
    int backwards;              // 1: the items in falling order
    int *status;
};

// An item is a run of seg_rows output rows of one strip of 128 columns.  Each
// CTA takes the items blockIdx.x, blockIdx.x + gridDim.x, ...; the input rows of
// its items (an item's output rows and one more at each end) follow one another
// through a ring of kRing row slots [plane][kPixRows][8 channels], each row one
// bulk copy per plane, so an input row is loaded once per item instead of once
// per output row (1.1 times for runs of 20 rows and more).
// An input row is also multiplied once: for each column offset dx and 16
// channels one MMA of N = 3 NOUT takes it (started dx pixels in: 8-pixel row
// groups 128 bytes apart (SBO), planes kPixRows * 16 bytes apart (LBO)) against
// the weights of its three row offsets, into the accumulators of the three
// output rows it belongs to, which lie side by side in a ring of kAccs blocks of
// NOUT tensor-memory columns (two MMAs where the ring wraps, and where a new
// row's accumulator starts from zero).  An output row still sums its taps in the
// order dy, dx, channel.  What bounds the MMAs is shared memory: A is 4 KB per
// 128 x K = 16 step whatever N is, and 40 cycles for N = 32 (4 + 1 KB at 128
// bytes per cycle, measured 39.6) against 57 for N = 96, so a row of a 32 -> 32
// layer takes about 400 cycles instead of 720.  The rest is the layer's
// activations in and out of HBM once a batch is larger than L2; consecutive
// layers walk the batch in opposite directions, so that a layer begins with what
// the one before wrote last.
// One thread issues the MMAs and another the copies, both ahead of the eight
// epilogue warps (two groups of four, an output row each).  The MMAs of a row are
// written out, their descriptors base plus constant: computed in a loop, an MMA
// took about 200 cycles to issue and the issuing thread set the pace (2600 cycles
// per row).
constexpr int kPixRows = 136;                        // staged pixels per row and plane (>= 130, multiple of 8)
constexpr int kChunkBytes = kPixRows * 16;           // 2176 = 17 x 128: every copy's destination 128-byte aligned
constexpr int kBoxPix = 130;                         // columns j0-1 .. j0+128
constexpr int kRing = 8;                             // row slots
constexpr int kAccs = 8;                             // accumulators: three being summed, the others being read
constexpr int kEpiGroups = 2;
constexpr int kConvThreads = 128 * kEpiGroups + 64;

// One contiguous copy global -> shared memory (16-byte aligned, a multiple of 16 bytes).
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

template <int CIN, int NOUT, int EPI>
__global__ void __launch_bounds__(kConvThreads) k_conv(ConvArgs a)
{
    constexpr int CH8 = CIN / 8;            // 16-byte planes per pixel
    constexpr int SLOT = CH8 * kChunkBytes;
    constexpr int KB = 3 * CIN;             // columns of the packed weights
    constexpr uint32_t WSBO = KB / 8 * 128;
    constexpr unsigned WBYTES = 3 * NOUT * KB * 2;
    constexpr int TCOLS = kAccs * NOUT;     // tensor-memory columns
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    unsigned char *sb = sm_raw + kRing * SLOT;   // the packed weights
    __shared__ __align__(8) uint64_t bar_row[kRing], bar_mma[kAccs], bar_free[kAccs], bar_w;
    __shared__ uint32_t tbase;
    __shared__ float s_bias[32];
    const int t = threadIdx.x, warp = t >> 5;
    const int items = a.count * a.tiles * a.segs;
    const int pitch = act_pitch(a.nx);
    const long long n = (long long)a.ny * a.nx;

    if (warp == 0) tc_alloc(&tbase, TCOLS);
    if (t < 32) s_bias[t] = (EPI == EPI_RELU || (EPI == EPI_LAST && t == 0)) ? a.bias[t] : 0.0f;   // LAST: one bias
    if (t == 0) {
        for (int k = 0; k < kRing; ++k) mbar_init(&bar_row[k], 1);
        for (int k = 0; k < kAccs; ++k) {
            mbar_init(&bar_mma[k], 1);
            mbar_init(&bar_free[k], 4);   // one arrival per warp of the group that reads it
        }
        mbar_init(&bar_w, 1);
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tbase;

    // item -> image, strip, first output row, output rows
    auto item_pos = [&](int it, int &img, int &jb, int &i0, int &rows) {
        if (a.backwards) it = items - 1 - it;
        const int strip = it / a.segs, seg = it - strip * a.segs;
        img = strip / a.tiles;
        jb = strip - img * a.tiles;
        i0 = seg * a.seg_rows;
        rows = min(a.seg_rows, a.ny - i0);
    };
    bool ok = true;
    if (warp == 4 * kEpiGroups + 1) {   // copies: the input rows of the CTA's items, a row per slot
        if ((t & 31) == 0 && (int)blockIdx.x < items) {
            // `produced` rows issued so far, the next one row pl (of p_rows + 2) of item p_it; `freed` rows no
            // longer read by any MMA
            int produced = 0, freed = 0, pl = 0, p_it = blockIdx.x;
            int p_img, p_jb, p_i0, p_rows;
            item_pos(p_it, p_img, p_jb, p_i0, p_rows);
            auto load_rows = [&]() {   // as many of the next input rows as there are free slots
                while (p_it < items && produced < freed + kRing) {
                    const int slot = produced % kRing, j0 = p_jb * kTile;
                    // the columns an output of this strip can read; what lies beyond is stale and feeds only
                    // outputs that are not stored
                    const unsigned bytes = 16u * (unsigned)min(kBoxPix, pitch - 8 - j0 + 2);
                    mbar_expect_tx(&bar_row[slot], CH8 * bytes);
                    const __nv_bfloat16 *src = a.in + (act_row(p_img, p_i0 + pl - 1, 0, CH8, a.ny, pitch) + j0 - 1) * 8;
#pragma unroll
                    for (int c8 = 0; c8 < CH8; ++c8)
                        bulk_load(sm_raw + slot * SLOT + c8 * kChunkBytes, src + (size_t)c8 * pitch * 8, bytes, &bar_row[slot]);
                    ++produced;
                    if (++pl == p_rows + 2) {
                        pl = 0;
                        p_it += gridDim.x;
                        if (p_it < items) item_pos(p_it, p_img, p_jb, p_i0, p_rows);
                    }
                }
            };
            mbar_expect_tx(&bar_w, WBYTES);
            bulk_load(sb, a.w, WBYTES, &bar_w);
            load_rows();
            // an output row's MMAs done: the input rows up to its last one are free.  (No barrier can run a
            // phase ahead of this thread: the next MMAs on it need rows that only this thread loads.)
            int g = 0, base_r = 0;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
                int img, jb, i0, rows;
                item_pos(it, img, jb, i0, rows);
                for (int q = 0; q < rows && ok; ++q, ++g) {
                    ok = mbar_wait(&bar_mma[g % kAccs], (g / kAccs) & 1);
                    freed = base_r + q + 3;
                    if (ok) load_rows();
                }
                base_r += rows + 2;
            }
            if (!ok) {   // bounded waits for the copies still in flight before their memory is released
                atomicExch(a.status, (int)SUPCG_ERR_TIMEOUT);
                (void)mbar_wait(&bar_w, 0);
                for (int r = max(0, produced - kRing); r < produced; ++r) (void)mbar_wait(&bar_row[r % kRing], (r / kRing) & 1);
            }
        }
        __syncwarp();
    } else if (warp == 4 * kEpiGroups) {   // MMAs
        if ((t & 31) == 0 && (int)blockIdx.x < items) {
            constexpr int STEPS = 3 * CH8 / 2;   // dx, then 16 channels
            constexpr uint32_t id1 = tc_idesc_bf16(128, NOUT), id2 = tc_idesc_bf16(128, 2 * NOUT), id3 = tc_idesc_bf16(128, 3 * NOUT);
            ok = mbar_wait(&bar_w, 0);
            const uint64_t w0 = tc_sdesc(smem_u32(sb), 128, WSBO);
            // the descriptors' address fields count 16 bytes
            auto ad = [](int step) { return (uint64_t)((2 * (step % (CH8 / 2)) * kChunkBytes + step / (CH8 / 2) * 16) / 16); };
            auto bd = [](int step, int s0) {
                return (uint64_t)((((step / (CH8 / 2)) * CH8 + 2 * (step % (CH8 / 2))) * 128 + s0 * NOUT / 8 * (int)WSBO) / 16);
            };
            bool issued = false;
            int base_o = 0, base_r = 0;   // the item's first output and input row, counted over the CTA's items
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
                int img, jb, i0, rows;
                item_pos(it, img, jb, i0, rows);
                for (int l = 0; l < rows + 2; ++l) {   // input row l meets the output rows l - 2 + s, s = 2 - dy
                    const int r = base_r + l, s_lo = max(0, 2 - l), s_hi = min(2, rows + 1 - l);
                    const int g0 = base_o + l - 2;     // the output row of s = 0
                    // a new output row: its accumulator's previous row read by the epilogue
                    if (s_hi == 2 && g0 + 2 >= kAccs) ok = mbar_wait(&bar_free[(g0 + 2) % kAccs], (((g0 + 2) / kAccs) - 1) & 1);
                    if (ok) ok = mbar_wait(&bar_row[r % kRing], (r / kRing) & 1);
                    if (!ok) break;
                    tc_fence_after();
                    issued = true;
                    const uint64_t a0 = tc_sdesc(smem_u32(sm_raw) + (uint32_t)((r % kRing) * SLOT), kChunkBytes, 128);
                    auto d_of = [&](int k) { return tmem + (uint32_t)(((g0 + k) % kAccs) * NOUT); };
                    if (s_lo == 0 && s_hi == 2) {
                        const uint32_t d0 = d_of(0), d1 = d_of(1), d2 = d_of(2);
                        tc_mma_bf16(d2, a0 + ad(0), w0 + bd(0, 2), id1, 0u);   // the new row starts from zero
                        if (d2 == d0 + 2 * NOUT) {
                            tc_mma_bf16(d0, a0 + ad(0), w0 + bd(0, 0), id2, 1u);
#pragma unroll
                            for (int k = 1; k < STEPS; ++k) tc_mma_bf16(d0, a0 + ad(k), w0 + bd(k, 0), id3, 1u);
                        } else if (d1 == 0 + tmem) {   // the ring starts over at the second row
                            tc_mma_bf16(d0, a0 + ad(0), w0 + bd(0, 0), id1, 1u);
                            tc_mma_bf16(d1, a0 + ad(0), w0 + bd(0, 1), id1, 1u);
#pragma unroll
                            for (int k = 1; k < STEPS; ++k) {
                                tc_mma_bf16(d0, a0 + ad(k), w0 + bd(k, 0), id1, 1u);
                                tc_mma_bf16(d1, a0 + ad(k), w0 + bd(k, 1), id2, 1u);
                            }
                        } else {                        // at the third
                            tc_mma_bf16(d0, a0 + ad(0), w0 + bd(0, 0), id2, 1u);
#pragma unroll
                            for (int k = 1; k < STEPS; ++k) {
                                tc_mma_bf16(d0, a0 + ad(k), w0 + bd(k, 0), id2, 1u);
                                tc_mma_bf16(d2, a0 + ad(k), w0 + bd(k, 2), id1, 1u);
                            }
                        }
                    } else {   // an item's first and last input rows: one output row at a time
#pragma unroll
                        for (int s0 = 0; s0 < 3; ++s0)
                            if (s0 >= s_lo && s0 <= s_hi)
#pragma unroll
                                for (int k = 0; k < STEPS; ++k)
                                    tc_mma_bf16(d_of(s0), a0 + ad(k), w0 + bd(k, s0), id1, (k > 0 || s0 < 2) ? 1u : 0u);
                    }
                    if (s_lo == 0) tc_commit(&bar_mma[g0 % kAccs]);   // the output row g0 ends here
                }
                base_o += rows;
                base_r += rows + 2;
            }
            if (!ok) {
                atomicExch(a.status, (int)SUPCG_ERR_TIMEOUT);
                if (issued) {   // a bounded wait for the MMAs in flight: the weights' barrier, in its second phase
                    tc_commit(&bar_w);
                    (void)mbar_wait(&bar_w, 1);
                }
            }
        }
        __syncwarp();
    } else {
        const int grp = warp >> 2;
        int o = 0;
        for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
            int img, jb, i0, rows;
            item_pos(it, img, jb, i0, rows);
            const int j = jb * kTile + (t & 127);
            const bool in = j < a.nx;
            for (int q = 0; q < rows; ++q, ++o) {
                if (o % kEpiGroups != grp) continue;
                const int acc_i = o % kAccs, i = i0 + q;
                __align__(16) __nv_bfloat16 mk[32];
                float res = 0.0f;
                if (in) {   // epilogue operands, fetched while the MMAs run
                    if (EPI == EPI_MASK)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            reinterpret_cast<uint4 *>(mk)[c] =
                                __ldg(reinterpret_cast<const uint4 *>(a.mask) + act_row(img, i, c, 4, a.ny, pitch) + j);
                    if (EPI == EPI_LAST) res = a.resid[img * n + (long long)i * a.nx + j] * a.rscale[3 * img + 1];
                }
                // (every lane polls; the vote keeps the warp together for the tensor-memory loads)
                ok = __all_sync(0xffffffffu, mbar_wait(&bar_mma[acc_i], (o / kAccs) & 1));
                if (!ok) break;
                tc_fence_after();
                float acc[32];
                const uint32_t lane_addr = tmem + (uint32_t)(NOUT * acc_i) + ((uint32_t)((warp & 3) * 32) << 16);
                tc_ld16(lane_addr, acc);
                if (NOUT == 32) tc_ld16(lane_addr + 16, acc + 16);
                tc_fence_before();
                __syncwarp();
                if ((t & 31) == 0) mbar_arrive(&bar_free[acc_i]);
                if (!in) continue;
                if (EPI == EPI_LAST) {
                    a.out_f[img * n + (long long)i * a.nx + j] = acc[0] + s_bias[0] + res;
                } else {
                    __align__(16) __nv_bfloat16 ob[32];
#pragma unroll
                    for (int c = 0; c < 32; ++c) {
                        float v = acc[c];
                        if (EPI == EPI_RELU) v = fmaxf(0.0f, v + s_bias[c]);
                        else v = (__bfloat162float(mk[c]) > 0.0f) ? v : 0.0f;
                        ob[c] = __float2bfloat16_rn(v);
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        *(reinterpret_cast<uint4 *>(a.out_bf) + act_row(img, i, c, 4, a.ny, pitch) + j) =
                            reinterpret_cast<const uint4 *>(ob)[c];
                }
            }
        }
        if (!ok && (t & 31) == 0) atomicExch(a.status, (int)SUPCG_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem, TCOLS);
}

template <int CIN, int NOUT, int EPI>
static int launch_conv(ConvArgs a, cudaStream_t st)
{
    constexpr int smem = kRing * (CIN / 8) * kChunkBytes + 9 * NOUT * CIN * 2;
    // attributes and the persistent grid size are per device
    static std::mutex mu;
    static int ctas_dev[kMaxDevices] = {};
    int dev = 0;
    int rc0 = current_device(&dev);
    if (rc0) return rc0;
    rc0 = func_attrs_once((const void *)k_conv<CIN, NOUT, EPI>, smem, (int)cudaSharedmemCarveoutMaxShared);
    if (rc0) return rc0;
    int ctas;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (!ctas_dev[dev]) {
            int nsm = 1;
            SUPCG_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
            int smem_sm = 0;
            SUPCG_CUDA_TRY(cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev));
            const int by_smem = smem_sm / (smem + 2048);   // dynamic + static shared memory and the per-CTA reserve
            // kAccs NOUT of the SM's 512 tensor-memory columns per CTA
            ctas_dev[dev] = nsm * std::max(1, std::min(by_smem, 512 / (kAccs * NOUT)));
        }
        ctas = ctas_dev[dev];
    }
    // rows per item: about one item per CTA, each item's two extra input rows being the cost of more, shorter ones
    a.tiles = (a.nx + kTile - 1) / kTile;
    const long long strips = (long long)a.count * a.tiles;
    const int per_strip = (int)std::max<long long>(1, std::min<long long>(a.ny, ctas / strips));
    a.seg_rows = (a.ny + per_strip - 1) / per_strip;
    a.segs = (a.ny + a.seg_rows - 1) / a.seg_rows;
    const unsigned grid = (unsigned)std::min<long long>(strips * a.segs, ctas);
    k_conv<CIN, NOUT, EPI><<<grid, kConvThreads, smem, st>>>(a);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

// ------------------------------------------------------------------ weight gradient
// dW[co][ci][dy][dx] = sum_p G[p][co] * in[p + (dy-1, dx-1)][ci],  db[co] = sum_p G[p][co].
// A contraction over pixels, on the tensor cores.  A tile is 128 columns of a pair of
// image rows i, i + 1: the four input rows i - 1 .. i + 2 and the two rows of G.  Per
// column offset dx one accumulator
//   D_dx[m][n] += sum_k A_dx[m][k] B[k][n],  m = (input row a, channel), n = (row b of G, channel)
// takes the tile's columns k; A_dx is the staged input started dx pixels in, and
// (a, b) is row offset dy = a - b, so that 6 of its 8 quarter blocks are wanted (the
// others are summed and not read).  Both operands are read MN-major from the stage
// layout [plane][columns][8 channels]: core matrices 128 bytes apart along the
// pixels (LBO), planes kWgA or kWgG bytes apart (SBO).  A tile arrives by two tensor
// copies, one of the four input rows and one of the two rows of G, in units of 8
// columns (128 bytes; the input from column j0 - 8 on): as 24 bulk copies, one per
// plane and row, the issuing thread needed 2500 cycles per tile and set the pace.  Shared memory bounds the MMAs (A is
// 4 KB per K = 16 step): N = 64 takes 48 cycles against 40 for the N = 32 of one row
// of G, and a pair stages six rows where two single rows staged eight, so a row of a
// 32 -> 32 layer takes about 780 cycles instead of 1220.  kWgStages stages keep three
// tiles of copies in flight (with two, one CTA waited for each tile's copies: 48 us for
// 32 x 128^2 against 26 us now).  db: four warps add the staged rows of G while the
// tensor core reads them.  Each persistent CTA (one per SM) writes one partial per row b
// of G; k_reduce sums the partials in order, so the result is deterministic.
constexpr int kWgStages = 4;
constexpr int kWgGroups = 18;                  // staged groups of 8 columns of the input: j0 - 8 .. j0 + 135
constexpr int kWgA = kWgGroups * 128;          // bytes of a staged plane of the input
constexpr int kWgG = kTile * 16;               // and of G
constexpr int kWgThreads = 192;   // four warps for db and the read-out, one that issues MMAs, one for the copies

// Bytes beyond the last stage that an MMA's A operand (16 planes from its stage's start) reads: rows of
// its accumulator that nothing reads
__host__ __device__ constexpr int wg_slack(int cin, int gch)
{
    const int over = 16 * kWgA - (4 * (cin / 8) * kWgA + 2 * (gch / 8) * kWgG);
    return over > 0 ? over : 0;
}

template <int CIN, int GCH>
__global__ void __launch_bounds__(kWgThreads) k_wgrad(int ny, int nx, int count, int cin_real, int cout, float *partial,
                                                      int *status, const __grid_constant__ CUtensorMap tin,
                                                      const __grid_constant__ CUtensorMap tg)
{
    constexpr int CH8 = CIN / 8, GH8 = GCH / 8, N = 2 * GCH;
    constexpr int STAGE = 4 * CH8 * kWgA + 2 * GH8 * kWgG;
    static_assert((kWgStages - 1) * STAGE + 16 * kWgA <= kWgStages * STAGE + wg_slack(CIN, GCH), "A's 16 planes lie in shared memory");
    constexpr int TCOLS = GCH == 32 ? 256 : 128;   // >= 3 N
    extern __shared__ __align__(1024) unsigned char sm_raw[];
    __shared__ __align__(8) uint64_t bar_tma[kWgStages], bar_mma[kWgStages], bar_g[kWgStages];
    __shared__ uint32_t tbase;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int tiles_row = (nx + kTile - 1) / kTile, pairs = (ny + 1) / 2, pitch = act_pitch(nx);
    const long long ntiles = (long long)count * pairs * tiles_row;
    const long long first = blockIdx.x, stride = gridDim.x;
    const int nq = first < ntiles ? (int)((ntiles - 1 - first) / stride) + 1 : 0;

    if (warp == 0) tc_alloc(&tbase, TCOLS);
    if (t == 0) {
        for (int k = 0; k < kWgStages; ++k) {
            mbar_init(&bar_tma[k], 1);
            mbar_init(&bar_mma[k], 1);
            mbar_init(&bar_g[k], GH8);   // one arrival per warp that reads G
        }
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tbase;

    // columns of tile q's contraction: a multiple of 16 (G is zero from nx on)
    auto tile_cols = [&](int q) {
        const int jb = (int)((first + (long long)q * stride) % tiles_row);
        return min(kTile, pitch - 8 - jb * kTile);
    };
    bool ok = true;
    float db[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) db[c] = 0.0f;
    if (warp == 5) {
        if (lane == 0) {
            for (int q = 0; q < nq; ++q) {   // tile q's rows into its stage, once the tile before it there is done
                const int buf = q % kWgStages;
                if (q >= kWgStages) {
                    const int ph = (q / kWgStages - 1) & 1;
                    ok = mbar_wait(&bar_mma[buf], ph) && mbar_wait(&bar_g[buf], ph);
                    if (!ok) {   // bounded waits for the copies still in flight before their memory is released
                        for (int k = q - kWgStages; k < q; ++k) (void)mbar_wait(&bar_tma[k % kWgStages], (k / kWgStages) & 1);
                        break;
                    }
                }
                const long long tile = first + (long long)q * stride;
                const long long rowid = tile / tiles_row;
                const int j0 = (int)(tile - rowid * tiles_row) * kTile;
                const int img = (int)(rowid / pairs), i = 2 * (int)(rowid - (long long)img * pairs);
                // rows are counted over the images, ny + 2 each, the first one row -1; what lies beyond the
                // tensor (columns, or the row after an odd last image) arrives as zeros
                const int row = img * (ny + 2) + i;
                const uint32_t st = smem_u32(sm_raw) + buf * STAGE, bar = smem_u32(&bar_tma[buf]);
                mbar_expect_tx(&bar_tma[buf], STAGE);
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                    " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(st),
                    "l"(reinterpret_cast<uint64_t>(&tin)), "r"(0), "r"(j0 / 8), "r"(0), "r"(row), "r"(bar)
                    : "memory");
                asm volatile(
                    "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                    " [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(st + 4 * CH8 * kWgA),
                    "l"(reinterpret_cast<uint64_t>(&tg)), "r"(0), "r"(j0 / 8 + 1), "r"(0), "r"(row + 1), "r"(bar)
                    : "memory");
            }
        }
        __syncwarp();
    } else if (warp == 4) {
        if (lane == 0 && nq > 0) {
            constexpr uint32_t idesc = tc_idesc_bf16(128, N) | (1u << 15) | (1u << 16);   // A and B MN-major
            int issued = 0;
            for (int q = 0; q < nq; ++q) {
                const int b = q % kWgStages;
                ok = mbar_wait(&bar_tma[b], (q / kWgStages) & 1);
                if (!ok) break;
                tc_fence_after();
                const uint32_t sa_u = smem_u32(sm_raw) + b * STAGE;
                // (column j0 - 1 is the input's eighth staged one)
                const uint64_t a0 = tc_sdesc(sa_u + 7 * 16, 128, kWgA), g0 = tc_sdesc(sa_u + 4 * CH8 * kWgA, 128, kWgG);
                const int ksteps = tile_cols(q) / 16;
                // (address fields count 16 bytes: a step of 16 pixels is 16 of them, a column offset one)
                if (ksteps == 8) {
#pragma unroll
                    for (int dx = 0; dx < 3; ++dx)
#pragma unroll
                        for (int ks = 0; ks < 8; ++ks)
                            tc_mma_bf16(tmem + (uint32_t)(dx * N), a0 + (uint64_t)(dx + 16 * ks), g0 + (uint64_t)(16 * ks), idesc,
                                        (q > 0 || ks > 0) ? 1u : 0u);
                } else {
                    for (int ks = 0; ks < ksteps; ++ks)
#pragma unroll
                        for (int dx = 0; dx < 3; ++dx)
                            tc_mma_bf16(tmem + (uint32_t)(dx * N), a0 + (uint64_t)(dx + 16 * ks), g0 + (uint64_t)(16 * ks), idesc,
                                        (q > 0 || ks > 0) ? 1u : 0u);
                }
                tc_commit(&bar_mma[b]);
                issued = q + 1;
            }
            // the last tile's MMAs complete after all earlier ones (commit order); after a timeout the wait is
            // for what is still in flight before its memory is released
            if (issued > 0) ok = mbar_wait(&bar_mma[(issued - 1) % kWgStages], ((issued - 1) / kWgStages) & 1) && ok;
        }
        __syncwarp();
    } else if (warp < GH8) {   // this warp's plane of G: 8 channels
        for (int q = 0; q < nq; ++q) {
            const int b = q % kWgStages, cols = tile_cols(q);
            ok = __all_sync(0xffffffffu, mbar_wait(&bar_tma[b], (q / kWgStages) & 1));
            if (!ok) break;
            const unsigned char *st = sm_raw + b * STAGE + 4 * CH8 * kWgA + warp * kWgG;
#pragma unroll
            for (int r = 0; r < 2; ++r)
                for (int k = lane; k < cols; k += 32) {
                    __align__(16) __nv_bfloat16 g[8];
                    *reinterpret_cast<uint4 *>(g) = *reinterpret_cast<const uint4 *>(st + r * GH8 * kWgG + k * 16);
#pragma unroll
                    for (int c = 0; c < 8; ++c) db[c] += __bfloat162float(g[c]);
                }
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_g[b]);
        }
    }
    if (!ok && lane == 0) atomicExch(status, (int)SUPCG_ERR_TIMEOUT);
    ok = __syncthreads_and(ok);
    tc_fence_after();
    if (ok && nq > 0 && warp < 4) {
        // lane m: plane m / 8 (input row a = plane / CH8, channel (plane % CH8) * 8 + m % 8).  A partial is
        // [dx][co][dy][ci], then db: consecutive lanes write consecutive ci
        const int m = warp * 32 + lane, a = (m >> 3) / CH8, ci = ((m >> 3) % CH8) * 8 + (m & 7);
        const int len = cout * cin_real * 9 + cout;
        const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
        for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                float acc[GCH];
#pragma unroll
                for (int c = 0; c < GCH; c += 16) tc_ld16(lane_addr + (uint32_t)(dx * N + b * GCH + c), acc + c);
                const int dy = a - b;
                float *out = partial + (size_t)(2 * blockIdx.x + b) * len;
                if (a < 4 && dy >= 0 && dy < 3 && ci < cin_real)
#pragma unroll
                    for (int co = 0; co < GCH; ++co)
                        if (co < cout) out[((dx * cout + co) * 3 + dy) * cin_real + ci] = acc[co];
            }
        float *dbo = partial + (size_t)(2 * blockIdx.x) * len + cout * cin_real * 9;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            float v = db[c];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0 && warp < GH8 && warp * 8 + c < cout) {
                dbo[warp * 8 + c] = v;
                dbo[len + warp * 8 + c] = 0.0f;   // the second partial has no part of db
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tc_dealloc(tmem, TCOLS);
}

constexpr int kWgradPartials = 2;   // partials per CTA (one CTA per SM)

// 4-D map of an activation tensor (groups of 8 columns, planes, rows of all images) with a box of
// `groups` groups x all planes x `rows` rows.
static int act_map(CUtensorMap *m, const __nv_bfloat16 *base, int ch, int ny, int nx, int count, int groups, int rows)
{
    const int pitch = act_pitch(nx);
    const cuuint64_t dims[4] = {64, (cuuint64_t)(pitch / 8), (cuuint64_t)(ch / 8), (cuuint64_t)count * (ny + 2)};
    const cuuint64_t strides[3] = {128, (cuuint64_t)pitch * 16, (cuuint64_t)(ch / 8) * pitch * 16};
    const cuuint32_t box[4] = {64, (cuuint32_t)groups, (cuuint32_t)(ch / 8), (cuuint32_t)rows};
    return encode_tiled(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16 *>(base), dims, strides, box);
}

// Weight gradient of one layer into partial[2 grid][len]; returns the partial count or an error (< 0).
template <int CIN, int GCH>
static int launch_wgrad(const __nv_bfloat16 *in, const __nv_bfloat16 *G, int cin_real, int cout, int ny, int nx,
                        int count, int max_ctas, float *partial, int *status, cudaStream_t st)
{
    constexpr int smem = kWgStages * (4 * (CIN / 8) * kWgA + 2 * (GCH / 8) * kWgG) + wg_slack(CIN, GCH);
    const int rc0 = func_attrs_once((const void *)k_wgrad<CIN, GCH>, smem, (int)cudaSharedmemCarveoutMaxShared);
    if (rc0) return rc0;
    const long long tiles = (long long)count * ((ny + 1) / 2) * ((nx + kTile - 1) / kTile);
    const int grid = (int)std::min<long long>(tiles, max_ctas);
    CUtensorMap tin, tg;
    int rc = act_map(&tin, in, CIN, ny, nx, count, kWgGroups, 4);
    if (!rc) rc = act_map(&tg, G, GCH, ny, nx, count, kTile / 8, 2);
    if (rc) return rc;
    k_wgrad<CIN, GCH><<<grid, kWgThreads, smem, st>>>(ny, nx, count, cin_real, cout, partial, status, tin, tg);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return kWgradPartials * grid;
}

// The layers' gradients from their partials, all layers in one launch.  A layer's gradient is
// out[co][ci][dy][dx], then db: element e of the partials' order [dx][co][dy][ci] is
// sum_b partial[b][e] in a fixed order: warp w of a block adds the partials b = w, w + 8, ...
// for 32 consecutive e (lane = e), then warp 0 adds the eight warp sums in warp order.  Eight
// loads in flight and sums in three FP32 parts (no less accurate than FP64 ones, on the FP32 pipe): with
// FP64 adds, one load at a time and a launch per layer the five layers took 65 us (32 x 128^2), 11 us now.
struct ReduceArgs {
    const float *partial[kCnnLayers];
    float *out[kCnnLayers];
    int nb[kCnnLayers], cout[kCnnLayers], cin[kCnnLayers], first[kCnnLayers];   // first: the layer's first block
};

__global__ void __launch_bounds__(256) k_reduce(ReduceArgs a)
{
    __shared__ float sh[3][8][32];
    int l = kCnnLayers - 1;
    while (l > 0 && (int)blockIdx.x < a.first[l]) --l;
    const float *partial = a.partial[l];
    const int nb = a.nb[l], cout = a.cout[l], cin = a.cin[l];
    const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
    const int e = (blockIdx.x - a.first[l]) * 32 + ln, len = cout * cin * 9 + cout;
    tf s = tf_make();
    if (e < len) {
        int b = w;
        for (; b + 56 < nb; b += 64) {
            float v[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = partial[(size_t)(b + 8 * k) * len + e];
#pragma unroll
            for (int k = 0; k < 8; ++k) tf_acc(s, v[k]);
        }
        for (; b < nb; b += 8) tf_acc(s, partial[(size_t)b * len + e]);
    }
    sh[0][w][ln] = s.h;
    sh[1][w][ln] = s.l;
    sh[2][w][ln] = s.m;
    __syncthreads();
    if (w == 0 && e < len) {
        tf sum = tf_make();
#pragma unroll
        for (int k = 0; k < 8; ++k) tf_add(sum, sh[0][k][ln], sh[1][k][ln], sh[2][k][ln]);
        float tot = (float)tf_to_double(sum);
        if (!isfinite(tot)) {   // an infinite partial (its TwoSum error is NaN): the plain sum
            double v = 0.0;
            for (int b = 0; b < nb; ++b) v += (double)partial[(size_t)b * len + e];
            tot = (float)v;
        }
        int o = e;
        if (e < 9 * cout * cin) {
            const int r = e / cin, ci = e - r * cin, dy = r % 3, co = (r / 3) % cout, dx = r / (3 * cout);
            o = (co * cin + ci) * 9 + dy * 3 + dx;
        }
        a.out[l][o] = tot;
    }
}

// ------------------------------------------------------------------ input, loss, optimiser
// Per-image unit-RMS scale factors sqrt(n / sum v^2) of x, tbar and (tg not null) the target
// (0 for an all-zero image): scale[3 img + k].  Grid (nblk, count, arrays), nblk =
// norm_blocks(n) <= kNormBlocks: each block sums a contiguous part of one image (exact
// products, sums in three FP32 parts: with FP64 ones the narrow pipe held this at 31 us for
// 8 x 512^2, 20 us now); the image's last block adds the partials in a fixed order and
// writes the FP32 factor.
constexpr int kNormBlocks = 256;
constexpr int kNormUnroll = 8;   // elements per thread in flight

// s += v^2: exactly where v^2 and its rounding error are FP32 numbers, else into the FP64 sum
// `rest` (*any then); their total over the block, in thread 0
__device__ __forceinline__ void sq_acc(tf &s, double &rest, bool &any, float v)
{
    const float a = fabsf(v);
    if (v == 0.0f || (a > 1e-15f && a < 1e15f)) {
        tf_acc_sq(s, v);
    } else {
        rest += (double)v * (double)v;
        any = true;
    }
}
__device__ __forceinline__ double sq_total(tf s, double rest, bool any, double *red)
{
    tf_warp_sum(s);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    float *f = reinterpret_cast<float *>(red);   // [8 warps][3]
    if (l == 0) {
        f[3 * w] = s.h;
        f[3 * w + 1] = s.l;
        f[3 * w + 2] = s.m;
    }
    __syncthreads();
    double v = 0.0;
    if (w == 0) {
        s = l < 8 ? tf{f[3 * l], f[3 * l + 1], f[3 * l + 2]} : tf_make();
        tf_warp_sum(s);
        if (l == 0) v = tf_to_double(s);
    }
    return __syncthreads_or(any) ? v + block_sum<256>(rest, red) : v;
}

static int norm_blocks(long long n) { return (int)std::max(1ll, std::min<long long>(kNormBlocks, n / 2048)); }

__global__ void __launch_bounds__(256) k_norms(const float *x, const float *tb, const float *tg, long long n, double *part,
                                               unsigned *counter, float *scale)
{
    __shared__ __align__(16) double red[40];
    __shared__ int sh_last;
    const int blk = blockIdx.x, nblk = gridDim.x, which = blockIdx.z, sum = 3 * blockIdx.y + which;
    const long long per = (n + nblk - 1) / nblk;
    const long long e0 = blk * per, e1 = e0 + per < n ? e0 + per : n;
    const float *vi = (which == 0 ? x : (which == 1 ? tb : tg)) + blockIdx.y * n;
    tf s = tf_make();
    double rest = 0.0;
    bool any = false;
    for (long long e = e0 + threadIdx.x; e < e1; e += 256 * kNormUnroll) {
        float v[kNormUnroll];
#pragma unroll
        for (int k = 0; k < kNormUnroll; ++k) v[k] = e + 256 * k < e1 ? vi[e + 256 * k] : 0.0f;
#pragma unroll
        for (int k = 0; k < kNormUnroll; ++k) sq_acc(s, rest, any, v[k]);
    }
    const double bs = sq_total(s, rest, any, red);
    if (threadIdx.x == 0) part[sum * kNormBlocks + blk] = bs;
    if (!last_block(&counter[sum], nblk, &sh_last)) return;
    if (threadIdx.x < 32) {
        const double *pp = part + sum * kNormBlocks;
        double tot = 0.0;
        for (int k = threadIdx.x; k < nblk; k += 32) tot += __ldcg(pp + k);
        tot = warp_sum(tot);
        if (threadIdx.x == 0) {
            scale[sum] = tot > 0.0 ? (float)sqrt((double)n / tot) : 0.0f;
            counter[sum] = 0;   // ready for the next launch
        }
    }
}

// Input tensor: channel 0 = x / rms(x), channel 1 = tbar scaled to unit RMS, channels 2..7 = 0 (the
// second plane, channels 8..15, is zero from its creation on).
__global__ void __launch_bounds__(256) k_pack_input(const float *x, const float *tb, const float *scale, int ny, int nx,
                                                    unsigned total, __nv_bfloat16 *act0)
{
    const unsigned p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= total) return;
    const unsigned row = p / (unsigned)nx, j = p - row * (unsigned)nx;
    const unsigned img = row / (unsigned)ny, i = row - img * (unsigned)ny;
    const float v0 = x[p] * scale[3 * img], v1 = tb[p] * scale[3 * img + 1];
    __align__(16) __nv_bfloat16 o[8];
    o[0] = __float2bfloat16_rn(v0);
    o[1] = __float2bfloat16_rn(v1);
#pragma unroll
    for (int c = 2; c < 8; ++c) o[c] = __float2bfloat16_rn(0.0f);
    *(reinterpret_cast<uint4 *>(act0) + act_row(img, i, 0, 2, ny, act_pitch(nx)) + j) = *reinterpret_cast<const uint4 *>(o);
}

// Loss L = mean (out - target~)^2 with target~ the target scaled per image to unit
// RMS (scale[3 img + 2]); G5 = dL/dout as a 16-channel BF16 tensor (channel 0; the second plane
// stays zero).  The last block adds the blocks' sums in a fixed order and writes L.
__global__ void __launch_bounds__(256) k_loss(const float *out, const float *target, const float *nscale, int ny, int nx,
                                              unsigned total, __nv_bfloat16 *G5, double *partial, unsigned *counter,
                                              double *loss)
{
    __shared__ __align__(16) double red[40];
    tf s = tf_make();
    double rest = 0.0;
    bool any = false;
    const float scale = (float)(2.0 / (double)total);
    const int pitch = act_pitch(nx);
    // (p < total + stride <= 2^31 + 2^18: no wrap)
    for (unsigned p = blockIdx.x * blockDim.x + threadIdx.x; p < total; p += gridDim.x * blockDim.x) {
        const unsigned row = p / (unsigned)nx, j = p - row * (unsigned)nx;
        const unsigned img = row / (unsigned)ny, i = row - img * (unsigned)ny;
        const float d = out[p] - target[p] * nscale[3 * img + 2];
        sq_acc(s, rest, any, d);
        __align__(16) __nv_bfloat16 o[8];
        o[0] = __float2bfloat16_rn(scale * d);
#pragma unroll
        for (int c = 1; c < 8; ++c) o[c] = __float2bfloat16_rn(0.0f);
        *(reinterpret_cast<uint4 *>(G5) + act_row(img, i, 0, 2, ny, pitch) + j) = *reinterpret_cast<const uint4 *>(o);
    }
    const double bs = sq_total(s, rest, any, red);
    __shared__ int sh_last;
    if (threadIdx.x == 0) partial[blockIdx.x] = bs;
    if (!last_block(counter, gridDim.x, &sh_last)) return;
    const double tot = block_sum_array<256>(partial, gridDim.x, red);
    if (threadIdx.x == 0) {
        *loss = tot / (double)total;
        *counter = 0;   // ready for the next launch
    }
}

// Adam on the FP32 master parameters.
__global__ void k_adam(float *w, const float *g, float *m, float *v, int len, float lr, float b1, float b2,
                       float c1, float c2, float eps)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= len) return;
    const float gg = g[e];
    const float mm = b1 * m[e] + (1.0f - b1) * gg;
    const float vv = b2 * v[e] + (1.0f - b2) * gg * gg;
    m[e] = mm;
    v[e] = vv;
    w[e] -= lr * (mm / c1) / (sqrtf(vv / c2) + eps);
}

// Packed BF16 GEMM weights of layer l (forward) and of its input-gradient pass,
// as GEMM B operands: row (2 - dy) NOUT + output channel, column dx * channels + channel,
// so that the rows of one dx and 16 channels are the N = 3 NOUT of one MMA:
//   fwd: B[(2 - dy) nout + co][dx cin + ci] = W[co][ci][dy][dx]          (co < cout, ci < cin_real; else 0)
//   bwd: B[(2 - dy) 32 + ci][dx gch + co]   = W[co][ci][2 - dy][2 - dx]  (flipped kernel, transposed channels)
// stored in the tensor cores' K-major core-matrix order (8 rows x 16 bytes per
// 128-byte block, blocks K-contiguous): element (row, k) at
// ((row / 8) * (K / 8) + k / 8) * 64 + (row % 8) * 8 + k % 8, so that one bulk
// copy puts it in shared memory ready for the MMA descriptors.
__device__ __forceinline__ int core_matrix_index(int row, int k, int K)
{
    return ((row >> 3) * (K >> 3) + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7);
}

__global__ void k_pack_weights(const float *W, int cout, int cin, int cin_real, int nout, __nv_bfloat16 *fwd, int gch,
                               __nv_bfloat16 *bwd)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < 9 * nout * cin) {
        const int row = e / (3 * cin), k = e - row * 3 * cin;
        const int dy = 2 - row / nout, co = row % nout, dx = k / cin, ci = k - dx * cin;
        const float v = (co < cout && ci < cin_real) ? W[(co * cin_real + ci) * 9 + dy * 3 + dx] : 0.0f;
        fwd[core_matrix_index(row, k, 3 * cin)] = __float2bfloat16_rn(v);
    }
    if (bwd && e < 9 * kCh * gch) {
        const int row = e / (3 * gch), k = e - row * 3 * gch;
        const int dy = 2 - row / kCh, ci = row % kCh, dx = k / gch, co = k - dx * gch;
        const float v = (ci < cin_real && co < cout) ? W[(co * cin_real + ci) * 9 + 8 - (dy * 3 + dx)] : 0.0f;
        bwd[core_matrix_index(row, k, 3 * gch)] = __float2bfloat16_rn(v);
    }
}

} // namespace supcg

// ------------------------------------------------------------------ network object
using namespace supcg;

static unsigned long long next_cnn_id()
{
    static std::atomic<unsigned long long> last{0};
    return ++last;
}

struct supcg_cnn_s {
    const unsigned long long id = next_cnn_id();
    int ny, nx, cap;             // image size and the largest batch the buffers hold
    int nparam;
    int off_w[kCnnLayers], off_b[kCnnLayers];
    float *params = nullptr, *grads = nullptr, *adam_m = nullptr, *adam_v = nullptr;
    __nv_bfloat16 *wf[kCnnLayers] = {}, *wb[kCnnLayers] = {};
    __nv_bfloat16 *act[kCnnLayers] = {};   // act[0] input (16 ch), act[1..4] hidden (32 ch)
    // gbuf[4] = dL/dout (16 ch); gbuf[l] = dL/dz of layer l's output (32 ch), in two buffers by turns: the backward
    // pass is done with gbuf[l] when gbuf[l - 2] is written
    __nv_bfloat16 *gbuf[kCnnLayers] = {};
    float *out = nullptr, *partial[kCnnLayers] = {};   // partial: the layers' weight-gradient partials
    float *scales = nullptr;      // per image: factors of x, tbar and the target to unit RMS
    double *npart = nullptr, *lpart = nullptr;
    unsigned *ncount = nullptr;
    struct Result {               // read back together
        double loss;
        int status;
    } *result = nullptr;
    int wg_ctas = 1;              // weight-gradient CTAs per layer
    long long step = 0;
    std::vector<void *> allocs;
};
typedef supcg_cnn_s *supcg_cnn;

static int cnn_alloc(supcg_cnn net, void **p, size_t bytes)
{
    if (cudaMalloc(p, bytes) != cudaSuccess) return SUPCG_ERR_NOMEM;
    net->allocs.push_back(*p);
    if (cudaMemset(*p, 0, bytes) != cudaSuccess) return SUPCG_ERR_CUDA;
    return SUPCG_OK;
}

static int cnn_pack(supcg_cnn net, cudaStream_t st)
{
    for (int l = 0; l < kCnnLayers; ++l) {
        const int gch = (l == kCnnLayers - 1) ? kInCh : kCh;   // channels of dL/dz_l as stored
        const int len = 9 * std::max(l_nout(l) * l_cin(l), kCh * gch);
        k_pack_weights<<<(len + 255) / 256, 256, 0, st>>>(net->params + net->off_w[l], l_cout(l), l_cin(l), l_cin_real(l),
                                                          l_nout(l), net->wf[l], gch, l > 0 ? net->wb[l] : nullptr);
    }
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

extern "C" int supcg_cnn_create(int ny, int nx, int max_batch, unsigned long long seed, supcg_cnn *out)
{
    if (!out || ny < 1 || nx < 1 || max_batch < 1 || max_batch > 65535 || (long long)ny * nx * max_batch > (1ll << 31))
        return SUPCG_ERR_ARG;
    *out = nullptr;
    auto *net = new (std::nothrow) supcg_cnn_s();
    if (!net) return SUPCG_ERR_NOMEM;
    net->ny = ny;
    net->nx = nx;
    net->cap = max_batch;
    int off = 0;
    for (int l = 0; l < kCnnLayers; ++l) {
        net->off_w[l] = off;
        off += l_cout(l) * l_cin_real(l) * 9;
        net->off_b[l] = off;
        off += l_cout(l);
    }
    net->nparam = off;
    // He-uniform initial weights from a seeded generator; the last layer starts at zero so that the
    // untrained network returns the plain nonascending direction.
    std::vector<float> h(off, 0.0f);
    unsigned long long s = seed ? seed : 0x9E3779B97F4A7C15ull;
    auto rnd = [&s]() {   // splitmix64
        s += 0x9E3779B97F4A7C15ull;
        unsigned long long z = s;
        z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
        z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
        z ^= z >> 31;
        return (double)(z >> 11) / 9007199254740992.0;
    };
    for (int l = 0; l + 1 < kCnnLayers; ++l) {
        const double lim = sqrt(6.0 / (9.0 * l_cin_real(l)));
        for (int e = 0; e < l_cout(l) * l_cin_real(l) * 9; ++e) h[net->off_w[l] + e] = (float)((2.0 * rnd() - 1.0) * lim);
    }
    const long long npix = (long long)ny * nx * max_batch;
    int rc = SUPCG_OK;
    rc = rc ? rc : cnn_alloc(net, (void **)&net->params, sizeof(float) * off);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->grads, sizeof(float) * off);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->adam_m, sizeof(float) * off);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->adam_v, sizeof(float) * off);
    for (int l = 0; l < kCnnLayers && !rc; ++l) {
        rc = cnn_alloc(net, (void **)&net->wf[l], 2 * (size_t)l_nout(l) * 9 * l_cin(l));
        if (!rc && l > 0) rc = cnn_alloc(net, (void **)&net->wb[l], 2 * (size_t)kCh * 9 * (l == kCnnLayers - 1 ? kInCh : kCh));
        // (a row more, which the last pair of an odd image's rows reads, and 64 elements: a row's copy ends
        // one column after the last plane)
        const size_t cols = ((size_t)max_batch * (ny + 2) + 1) * act_pitch(nx);
        if (!rc) rc = cnn_alloc(net, (void **)&net->act[l], 2 * (cols * (l == 0 ? kInCh : kCh) + 64));
        const int last = l == kCnnLayers - 1;
        if (!rc && (l < 2 || last)) rc = cnn_alloc(net, (void **)&net->gbuf[l], 2 * (cols * (last ? kInCh : kCh) + 64));
        if (l >= 2 && !last) net->gbuf[l] = net->gbuf[l - 2];
    }
    int dev = 0, nsm = 1;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        rc = SUPCG_ERR_CUDA;
    net->wg_ctas = nsm;
    for (int l = 0; l < kCnnLayers && !rc; ++l)
        rc = cnn_alloc(net, (void **)&net->partial[l],
                       sizeof(float) * net->wg_ctas * kWgradPartials * (l_cout(l) * l_cin_real(l) * 9 + l_cout(l)));
    rc = rc ? rc : cnn_alloc(net, (void **)&net->out, sizeof(float) * npix);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->scales, sizeof(float) * 3 * max_batch);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->npart, sizeof(double) * 3 * kNormBlocks * max_batch);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->ncount, sizeof(unsigned) * (3 * max_batch + 1));   // the last: k_loss
    rc = rc ? rc : cnn_alloc(net, (void **)&net->lpart, sizeof(double) * 1024);
    rc = rc ? rc : cnn_alloc(net, (void **)&net->result, sizeof(supcg_cnn_s::Result));
    if (!rc && cudaMemcpy(net->params, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice) != cudaSuccess)
        rc = SUPCG_ERR_CUDA;
    if (!rc) rc = cnn_pack(net, 0);
    if (!rc && cudaDeviceSynchronize() != cudaSuccess) rc = SUPCG_ERR_CUDA;
    if (rc) {
        for (void *p : net->allocs) cudaFree(p);
        delete net;
        return rc;
    }
    *out = net;
    return SUPCG_OK;
}

extern "C" int supcg_cnn_destroy(supcg_cnn net)
{
    if (!net) return SUPCG_ERR_ARG;
    cudaDeviceSynchronize();
    for (void *p : net->allocs) cudaFree(p);
    delete net;
    return SUPCG_OK;
}

extern "C" int supcg_cnn_num_params(supcg_cnn net) { return net ? net->nparam : SUPCG_ERR_ARG; }

// Host copy of all FP32 parameters: for each layer W[cout][cin][3][3] then b[cout].
extern "C" int supcg_cnn_get_params(supcg_cnn net, float *h_params)
{
    if (!net || !h_params) return SUPCG_ERR_ARG;
    SUPCG_CUDA_TRY(cudaMemcpy(h_params, net->params, sizeof(float) * net->nparam, cudaMemcpyDeviceToHost));
    return SUPCG_OK;
}

extern "C" int supcg_cnn_set_params(supcg_cnn net, const float *h_params)
{
    if (!net || !h_params) return SUPCG_ERR_ARG;
    SUPCG_CUDA_TRY(cudaMemcpy(net->params, h_params, sizeof(float) * net->nparam, cudaMemcpyHostToDevice));
    int rc = cnn_pack(net, 0);
    if (rc) return rc;
    SUPCG_CUDA_TRY(cudaDeviceSynchronize());
    return SUPCG_OK;
}

namespace supcg {

// Forward pass of `count` images: out[count][ny][nx] (FP32, unit-RMS scale); with a target, its scale
// factors too.
static int cnn_forward_t(supcg_cnn net, const float *d_x, const float *d_tbar, const float *d_target, int count, cudaStream_t st)
{
    const long long n = (long long)net->ny * net->nx;
    k_norms<<<dim3(norm_blocks(n), count, d_target ? 3 : 2), 256, 0, st>>>(d_x, d_tbar, d_target, n, net->npart, net->ncount,
                                                                          net->scales);
    k_pack_input<<<(unsigned)((n * count + 255) / 256), 256, 0, st>>>(d_x, d_tbar, net->scales, net->ny, net->nx,
                                                                     (unsigned)(n * count), net->act[0]);
    SUPCG_CUDA_TRY(cudaGetLastError());
    ConvArgs a = {};
    a.ny = net->ny;
    a.nx = net->nx;
    a.count = count;
    a.status = &net->result->status;
    int rc;
    for (int l = 0; l < kCnnLayers; ++l) {
        a.backwards = l & 1;
        a.in = net->act[l];
        a.w = net->wf[l];
        a.bias = net->params + net->off_b[l];
        if (l + 1 < kCnnLayers) {
            a.out_bf = net->act[l + 1];
            rc = (l == 0) ? launch_conv<kInCh, kCh, EPI_RELU>(a, st) : launch_conv<kCh, kCh, EPI_RELU>(a, st);
        } else {
            a.out_f = net->out;
            a.resid = d_tbar;
            a.rscale = net->scales;
            rc = launch_conv<kCh, 16, EPI_LAST>(a, st);
        }
        if (rc) return rc;
    }
    return SUPCG_OK;
}

// Backward pass after cnn_forward with dL/dout in gbuf[4]: gradients into net->grads.
static int cnn_backward(supcg_cnn net, int count, cudaStream_t st)
{
    ConvArgs a = {};
    a.ny = net->ny;
    a.nx = net->nx;
    a.count = count;
    a.status = &net->result->status;
    ReduceArgs ra = {};
    for (int l = kCnnLayers - 1; l >= 0; --l) {
        const int cin_real = l_cin_real(l), cout = l_cout(l);
        float *part = net->partial[l];
        ra.partial[l] = part;
        ra.out[l] = net->grads + net->off_w[l];
        ra.cout[l] = cout;
        ra.cin[l] = cin_real;
        // weight gradient of layer l: input act[l], output gradient gbuf[l]
        int nb;
        if (l == 0)
            nb = launch_wgrad<kInCh, kCh>(net->act[0], net->gbuf[0], cin_real, cout, net->ny, net->nx, count,
                                          net->wg_ctas, part, &net->result->status, st);
        else if (l == kCnnLayers - 1)
            nb = launch_wgrad<kCh, kInCh>(net->act[l], net->gbuf[l], cin_real, cout, net->ny, net->nx, count,
                                          net->wg_ctas, part, &net->result->status, st);
        else
            nb = launch_wgrad<kCh, kCh>(net->act[l], net->gbuf[l], cin_real, cout, net->ny, net->nx, count,
                                        net->wg_ctas, part, &net->result->status, st);
        if (nb < 0) return nb;
        ra.nb[l] = nb;
        if (l == 0) break;
        // input gradient: dL/dz_{l-1} = conv(gbuf[l], flipped W_l) masked by act[l] > 0
        a.backwards = l & 1;
        a.in = net->gbuf[l];
        a.w = net->wb[l];
        a.mask = net->act[l];
        a.out_bf = net->gbuf[l - 1];
        int rc = (l == kCnnLayers - 1) ? launch_conv<kInCh, kCh, EPI_MASK>(a, st) : launch_conv<kCh, kCh, EPI_MASK>(a, st);
        if (rc) return rc;
    }
    int blocks = 0;
    for (int l = 0; l < kCnnLayers; ++l) {
        ra.first[l] = blocks;
        blocks += (ra.cout[l] * ra.cin[l] * 9 + ra.cout[l] + 31) / 32;
    }
    k_reduce<<<blocks, 256, 0, st>>>(ra);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

// The loss and dL/dout in gbuf[4] after cnn_forward_t with the target.
static int cnn_loss(supcg_cnn net, const float *d_target, int count, cudaStream_t st)
{
    const long long total = (long long)net->ny * net->nx * count;
    const int blocks = (int)std::min<long long>(1024, (total + 255) / 256);
    k_loss<<<blocks, 256, 0, st>>>(net->out, d_target, net->scales, net->ny, net->nx, (unsigned)total,
                                  net->gbuf[kCnnLayers - 1], net->lpart, net->ncount + 3 * net->cap, &net->result->loss);
    SUPCG_CUDA_TRY(cudaGetLastError());
    return SUPCG_OK;
}

int cnn_forward(supcg_cnn net, const float *d_x, const float *d_tbar, int count, cudaStream_t st)
{
    return cnn_forward_t(net, d_x, d_tbar, nullptr, count, st);
}

} // namespace supcg

namespace supcg {
float *cnn_output(supcg_cnn net) { return net->out; }
unsigned long long cnn_id(supcg_cnn net) { return net->id; }
int cnn_shape(supcg_cnn net, int *ny, int *nx)
{
    *ny = net->ny;
    *nx = net->nx;
    return SUPCG_OK;
}
int cnn_capacity(supcg_cnn net, int *max_batch)
{
    *max_batch = net->cap;
    return SUPCG_OK;
}
} // namespace supcg

static int cnn_check(supcg_cnn net, int count)
{
    return (!net || count < 1 || count > net->cap) ? SUPCG_ERR_ARG : SUPCG_OK;
}

// Waits for the stream; the network's status, and the last loss into *h_loss (nullable).
static int cnn_status(supcg_cnn net, cudaStream_t st, double *h_loss = nullptr)
{
    supcg_cnn_s::Result r = {};
    SUPCG_CUDA_TRY(cudaMemcpyAsync(&r, net->result, sizeof(r), cudaMemcpyDeviceToHost, st));
    SUPCG_CUDA_TRY(cudaStreamSynchronize(st));
    if (h_loss) *h_loss = r.loss;
    return r.status;
}

extern "C" int supcg_cnn_forward(supcg_cnn net, const float *d_x, const float *d_tbar, int count, float *d_out,
                                 void *stream)
{
    int rc = cnn_check(net, count);
    if (rc || !d_x || !d_tbar || !d_out) return rc ? rc : SUPCG_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = cnn_forward(net, d_x, d_tbar, count, st))) return rc;
    SUPCG_CUDA_TRY(cudaMemcpyAsync(d_out, net->out, sizeof(float) * (size_t)net->ny * net->nx * count,
                                   cudaMemcpyDeviceToDevice, st));
    return cnn_status(net, st);
}

extern "C" int supcg_cnn_gradients(supcg_cnn net, const float *d_x, const float *d_tbar, const float *d_target,
                                   int count, float *h_grads, double *h_loss, void *stream)
{
    int rc = cnn_check(net, count);
    if (rc || !d_x || !d_tbar || !d_target || !h_grads) return rc ? rc : SUPCG_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = cnn_forward_t(net, d_x, d_tbar, d_target, count, st))) return rc;
    if ((rc = cnn_loss(net, d_target, count, st))) return rc;
    if ((rc = cnn_backward(net, count, st))) return rc;
    SUPCG_CUDA_TRY(cudaMemcpyAsync(h_grads, net->grads, sizeof(float) * net->nparam, cudaMemcpyDeviceToHost, st));
    return cnn_status(net, st, h_loss);
}

extern "C" int supcg_cnn_train_step(supcg_cnn net, const float *d_x, const float *d_tbar, const float *d_target,
                                    int count, double lr, double *h_loss, void *stream)
{
    int rc = cnn_check(net, count);
    if (rc || !d_x || !d_tbar || !d_target || !(lr > 0.0)) return rc ? rc : SUPCG_ERR_ARG;
    cudaStream_t st = (cudaStream_t)stream;
    if ((rc = cnn_forward_t(net, d_x, d_tbar, d_target, count, st))) return rc;
    if ((rc = cnn_loss(net, d_target, count, st))) return rc;
    if ((rc = cnn_backward(net, count, st))) return rc;
    net->step += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = (float)(1.0 - pow(0.9, (double)net->step)), c2 = (float)(1.0 - pow(0.999, (double)net->step));
    k_adam<<<(net->nparam + 255) / 256, 256, 0, st>>>(net->params, net->grads, net->adam_m, net->adam_v, net->nparam,
                                                      (float)lr, b1, b2, c1, c2, 1e-8f);
    SUPCG_CUDA_TRY(cudaGetLastError());
    if ((rc = cnn_pack(net, st))) return rc;
    return h_loss ? cnn_status(net, st, h_loss) : SUPCG_OK;
}
