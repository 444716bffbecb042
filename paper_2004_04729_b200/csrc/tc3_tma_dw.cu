// Weight gradient of 3x3 convolutions (stride 1, pad 1) on the tensor cores, both operands brought
// in by tiled copies (Eq. (qdw), "analogous for convolutional layers"):
//   dW[co][ci][ky][kx] = Delta * sum_(b,j) X[b][ci][j] * q[b][co][j - (ky-1) W - (kx-1)]
// with j a position of the image (row-major), the code taken as zero outside the image and where
// the column x - (kx-1) leaves the row.
//
// The reduction index is the position. The activations lie [b][ci][position], so 64 consecutive
// positions of 128 input channels are one K-major tile (A, M = input channels). The quantizer has
// written the codes position-major, [b][position][co] in bf16, so a run of positions of 64 output
// channels is one MN-major panel (B, N = output channels), one 128-byte row per position, and a
// tap is only a different start row of that panel (the 128-byte swizzle is a function of the
// shared-memory address). The copy engine zero-fills the rows before the first and after the last
// position of the image, which is the padding above and below. Left/right padding cannot be a row
// offset: a CTA handles ONE kernel column kx, and one warp zeroes, in the freshly copied panel, the
// rows of image column 0 (kx = 0) or W-1 (kx = 2) before the MMAs read it.
//
// Per CTA: a range of segments (runs of up to 512 positions of one image, with a halo of W+1 rows
// on either side), an output tile of 128 input channels x 64 or 128 output channels, the three
// taps ky of its kx as three accumulators in tensor memory. The three taps of 64 output channels
// share one MMA of N = 192, whose 64-column groups start W rows apart.
// fp32 activations are two bf16 pieces, one after the other along the batch. Layers of at most 64 input channels put both
// pieces of a position on the two halves of one tile (half as many MMAs, the codes are read once; 64 -> 64 at 32x32, batch
// 128: 100 -> 91 us for the whole call).
// Warp 0 copies code panels, warp 1 activation tiles, warp 2 issues the MMAs, warp 3 zeroes the
// masked rows, warps 4-7 stage the accumulators in shared memory and the copy engine adds them into a
// zero-initialised fp32 scratch [tap][co][ci] (the reduction over CTAs; the order of the additions,
// hence the last bits of dW, can differ from run to run). A second kernel scales by Delta, writes
// dW[co][ci][ky][kx] and puts the zeros back. Every wait is bounded.
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace tc;

constexpr int kThreadsW3 = 8 * 32;
constexpr int kXTile = 16384;             // [128 ci][64 positions] bf16
constexpr int kXS = 2;                    // most 64-position stages per activation slot (one hand-over)
constexpr int kMaxNX = 4;
constexpr int kMaxNQ = 3;                 // most code buffers

struct Dw3T {
    int Cout, W, HW;
    int code_batch;               // images of the code tensor (the activations may hold two pieces of every image, one after the other)
    int split;                    // both pieces of (at most 64) channels share a tile: rows 0-63 the high ones, 64-127 the low ones
    int SEG;                      // positions per segment (multiple of 64)
    int segs_per_img;
    long long nseg, per_split;
    int nsplit;
    int ci_tiles, co_tiles;
    int rows_box, nload;          // a panel is copied as nload boxes of rows_box rows
    int panel_bytes;              // multiple of 1024
    int nx, xs;                   // activation slots in flight, 64-position stages of one
    int nq;                       // code buffers in flight
    int stage_chunks;             // 32-column chunks of the accumulators that fit the shared memory at once
    int phase_tiles;              // > 0: a stride-2 layer on phase images, this many 128-channel tiles per phase (phase
                                  // ph = 2 py + px holds channels ph * 128 * phase_tiles ...). Only the taps with
                                  // ky in {1} (py = 0) or {0, 1} (py = 1), kx likewise, are wanted: the work items of
                                  // the other kernel columns do not exist and the other rows' MMAs are left out
    int *err_flag;
    unsigned long long *stats;    // wait counters (may be null)
};

struct PipeW3 {
    unsigned long long x_full[kMaxNX], x_empty[kMaxNX], q_full[kMaxNQ], q_ready[kMaxNQ], q_empty[kMaxNQ], acc;
    unsigned tmem_base;
};

// NP: 64-channel panels of the code operand (N = 64 NP output channels per tap)
template <int NP>
__global__ void __launch_bounds__(kThreadsW3, 1)
tc3_tma_dw_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_x,
                  const __grid_constant__ CUtensorMap map_acc, const Dw3T p) {
    constexpr int TCOLS = NP == 2 ? 512 : 256;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *x_s = smem;                                   // nx activation slots
    const int x_slot = p.xs * kXTile;
    unsigned char *q_s = x_s + p.nx * x_slot;                    // nq buffers x NP panels
    const int qbuf_bytes = NP * p.panel_bytes;
    __shared__ PipeW3 pipe;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    // work item: (output tile, kernel column, range of segments)
    const int split = blockIdx.x % p.nsplit;
    int rest = blockIdx.x / p.nsplit;
    int kx, ci_t, co_t, live_lo = 0;                    // phase images: taps ky = live_lo .. 1 are accumulated (NP == 2)
    int c_lo = 0, c_hi = (NP == 2 ? 384 : 192) / 32;    // 32-column chunks of the accumulators that are handed over
    if (p.phase_tiles > 0) {
        // per output-channel tile: the phases in order, one kernel column (kx = 1) per channel tile of a phase with
        // px = 0, two (kx = 0, 1) with px = 1
        const int tp = p.phase_tiles, per_co = 6 * tp;
        co_t = rest / per_co;
        int r = rest - co_t * per_co;
        const int py = r / (3 * tp);
        r -= py * 3 * tp;
        if (r < tp) { ci_t = 2 * py * tp + r; kx = 1; }
        else { r -= tp; ci_t = (2 * py + 1) * tp + (r >> 1); kx = r & 1; }
        // NP == 2: columns 0-127 are ky = 0, 128-255 ky = 1; NP == 1: 0-63 ky = 2, 64-127 ky = 1, 128-191 ky = 0
        if (NP == 2) { live_lo = py ? 0 : 1; c_lo = 4 * live_lo; c_hi = 8; }
        else { c_lo = 2; c_hi = py ? 6 : 4; }
    } else {
        kx = rest % 3;
        rest /= 3;
        ci_t = rest % p.ci_tiles;
        co_t = rest / p.ci_tiles;
    }
    const int ci0 = ci_t * 128;
    const int co0 = co_t * 64 * NP;
    const long long g0 = split * p.per_split;
    const long long g1 = g0 + p.per_split < p.nseg ? g0 + p.per_split : p.nseg;
    const int halo = p.W + 1;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxNX; ++s) { mbar_init(&pipe.x_full[s], 1); mbar_init(&pipe.x_empty[s], 1); }
        for (int s = 0; s < kMaxNQ; ++s) { mbar_init(&pipe.q_full[s], 1); mbar_init(&pipe.q_ready[s], 1); mbar_init(&pipe.q_empty[s], 1); }
        mbar_init(&pipe.acc, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_x);
        tma_prefetch_desc(&map_acc);
    }
    if (warp == 2) tmem_alloc(&pipe.tmem_base, TCOLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = pipe.tmem_base;
    chain_wait();        // from here on the kernel reads what earlier kernels wrote

    // a segment: image and first position; they are walked one after the other
    struct Seg { int b, u0; };
    auto first_seg = [&] {
        const int b = static_cast<int>(g0 / p.segs_per_img);
        return Seg{b, static_cast<int>(g0 - static_cast<long long>(b) * p.segs_per_img) * p.SEG};
    };
    auto next_seg = [&](Seg &s) {
        s.u0 += p.SEG;
        if (s.u0 >= p.HW) { s.u0 = 0; ++s.b; }
    };
    auto stages_of = [&](const Seg &s) {         // of 64 positions
        const int left = p.HW - s.u0;
        return ((left < p.SEG ? left : p.SEG) + 63) >> 6;
    };
    const int nseg = g1 > g0 ? static_cast<int>(g1 - g0) : 0;
    // The activation stages of this CTA are consecutive 64-position blocks of consecutive images; a
    // slot holds xs consecutive blocks of one image. A new slot starts at the CTA's first stage, at
    // the first block of an image, and after xs stages (copy and MMA threads follow the same rule).

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            const unsigned tx = static_cast<unsigned>(NP * p.nload * p.rows_box * 128);
            int buf = 0;
            unsigned parity = 1;                   // a fresh barrier passes a wait on the previous phase
            Seg sg = first_seg();
            long long waited = 0;
            for (int i = 0; i < nseg; ++i, next_seg(sg)) {
                ok = mbar_wait_timed(&pipe.q_empty[buf], parity, p.err_flag, waited);
                if (!ok) break;
                unsigned char *dst = q_s + buf * qbuf_bytes;
                mbar_expect_tx(&pipe.q_full[buf], tx);
#pragma unroll
                for (int pn = 0; pn < NP; ++pn)
                    for (int l = 0; l < p.nload; ++l)
                        tma_load_3d(dst + pn * p.panel_bytes + l * p.rows_box * 128, &map_q, co0 + 64 * pn,
                                    sg.u0 - halo + l * p.rows_box, sg.b % p.code_batch, &pipe.q_full[buf]);
                if (++buf == p.nq) { buf = 0; parity ^= 1u; }
            }
            report_wait(p.stats, 3, waited);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            bool ok = true;
            int s = 0, j = p.xs;                   // j: stages already in the current slot
            unsigned parity = 1;
            long long waited = 0;
            Seg sg = first_seg();
            for (int i = 0; i < nseg && ok; ++i, next_seg(sg)) {
                const int ns = stages_of(sg), b = sg.b;
                for (int k = 0; k < ns; ++k) {
                    const int blk = (sg.u0 >> 6) + k;
                    if (j == p.xs || blk == 0) {
                        ok = mbar_wait_timed(&pipe.x_empty[s], parity, p.err_flag, waited);
                        if (!ok) break;
                        unsigned char *dst = x_s + s * x_slot;
                        // blocks of the image that the slot takes; positions past the image's end read as zero
                        const int nx = p.HW - blk * 64 > 64 ? p.xs : 1;
                        mbar_expect_tx(&pipe.x_full[s], nx * kXTile);
#pragma unroll
                        for (int i = 0; i < kXS; ++i) {
                            if (i >= nx) break;
                            tma_load_3d(dst + i * kXTile, &map_x, (blk + i) * 64, ci0, b, &pipe.x_full[s]);
                            if (p.split)
                                tma_load_3d(dst + i * kXTile + kXTile / 2, &map_x, (blk + i) * 64, 0, b + p.code_batch, &pipe.x_full[s]);
                        }
                        if (++s == p.nx) { s = 0; parity ^= 1u; }
                        j = 0;
                    }
                    ++j;
                }
            }
            report_wait(p.stats, 4, waited);
        }
    } else if (warp == 2) {
        {   // the whole warp runs the loop (uniform control flow and operands); one elected lane issues
            // tap ky reads a panel from row (2 - ky) W + (2 - kx) on. The three taps of a panel share ONE MMA of N = 192 whose
            // 64-column groups start W rows apart (columns 0-63: ky = 2, 64-127: ky = 1, 128-191: ky = 0; the second panel's
            // behind them). An MMA of N columns takes max(N/2, 32 + N/4) clocks, 96 for one of 192 against 144 for three of 64;
            // and where three of N = 128 over both panels read 24 KB of shared memory per 16 positions, two of 192 read 20, beside
            // the 8 that the copies write: 128 bytes a clock is what there is (260 clocks per 16 positions where it was 290).
            // Phase images have one or two live taps: an MMA of N = 128 over both panels per tap (columns 128 ky ...).
            constexpr unsigned idesc128 = make_idesc(128, 128, false, true), idesc192 = make_idesc(128, 192, false, true);
            const bool phases = NP == 2 && p.phase_tiles > 0;
            const unsigned r0 = static_cast<unsigned>((2 * p.W + 2 - kx) * 8), r1 = static_cast<unsigned>((p.W + 2 - kx) * 8),
                           r2 = static_cast<unsigned>((2 - kx) * 8);     // start rows in 16-byte units
            bool ok = true;
            int slot = -1, j = p.xs, buf = 0;
            unsigned xpar = 0, qpar = 0;
            unsigned acc_on = 0u;
            Seg sg = first_seg();
            long long wq = 0, wx = 0;
            const long long born = clock64();
            for (int i = 0; i < nseg && ok; ++i, next_seg(sg)) {
                ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.q_ready[buf], qpar, p.err_flag, wq));
                if (!ok) break;
                tc_fence_after();
                const int u0 = sg.u0, ns = stages_of(sg);
                const unsigned q_addr = smem_u32(q_s + buf * qbuf_bytes);
                // the panels' three taps; in phase mode tap ky = 0 and tap ky = 1 of both panels
                const unsigned long long bA = phases ? make_desc(q_addr, p.panel_bytes, 1024) + r0 : make_desc(q_addr, p.W * 128, 1024) + r2;
                const unsigned long long bB = phases ? make_desc(q_addr, p.panel_bytes, 1024) + r1 : bA + (static_cast<unsigned>(p.panel_bytes) >> 4);
                for (int k = 0; k < ns && ok; ++k) {
                    const int blk = (u0 >> 6) + k;
                    if (j == p.xs || blk == 0) {
                        if (slot >= 0 && elect_one()) mma_commit(&pipe.x_empty[slot]);
                        if (++slot == p.nx) { slot = 0; xpar ^= 1u; }
                        ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.x_full[slot], xpar, p.err_flag, wx));
                        if (!ok) break;
                        tc_fence_after();
                        j = 0;
                    }
                    // the last stage of an image may hold fewer than 64 positions: skip the 16-position
                    // slices that are entirely zero fill
                    const int left = p.HW - (u0 + 64 * k);
                    const int nk = left >= 64 ? 4 : (left + 15) >> 4;
                    const unsigned long long ad = make_desc(smem_u32(x_s + slot * x_slot + j * kXTile), 16, 1024);
                    const unsigned radv = static_cast<unsigned>(64 * k * 8);
                    auto slice = [&](int kk, unsigned on) {
                        const unsigned adv = radv + kk * 128;                 // 16 rows = 2048 bytes
                        if (phases) {
                            if (live_lo == 0) mma_bf16(tmem_base, ad + 2 * kk, bA + adv, idesc128, on);
                            mma_bf16(tmem_base + 128, ad + 2 * kk, bB + adv, idesc128, on);
                        } else {
                            mma_bf16(tmem_base, ad + 2 * kk, bA + adv, idesc192, on);
                            if (NP == 2) mma_bf16(tmem_base + 192, ad + 2 * kk, bB + adv, idesc192, on);
                        }
                    };
                    if (elect_one()) {
                        slice(0, acc_on);
                        if (nk == 4) {
#pragma unroll
                            for (int kk = 1; kk < 4; ++kk) slice(kk, 1u);
                        } else {
                            for (int kk = 1; kk < nk; ++kk) slice(kk, 1u);
                        }
                    }
                    acc_on = 1u;
                    ++j;
                }
                if (ok && elect_one()) mma_commit(&pipe.q_empty[buf]);
                if (++buf == p.nq) { buf = 0; qpar ^= 1u; }
            }
            if (ok && slot >= 0 && elect_one()) mma_commit(&pipe.x_empty[slot]);
            if (ok && g1 > g0 && elect_one()) mma_commit(&pipe.acc);
            if (lane == 0) {
                report_wait(p.stats, 0, wq);
                report_wait(p.stats, 1, wx);
                report_wait(p.stats, 6, clock64() - born);
                report_wait(p.stats, 7, 1);
            }
        }
    } else if (warp == 3) {
        // masked rows: image column 0 for kx = 0, W-1 for kx = 2 (generic-proxy writes, then a proxy
        // fence so that the tensor core sees them)
        int buf = 0;
        unsigned parity = 0;
        const int zc = kx == 0 ? 0 : p.W - 1;
        const int rows_total = p.nload * p.rows_box;
        Seg sg = first_seg();
        for (int i = 0; i < nseg; ++i, next_seg(sg)) {
            if (!mbar_wait(&pipe.q_full[buf], parity, p.err_flag)) break;
            if (kx != 1) {
                unsigned char *qb = q_s + buf * qbuf_bytes;
                const int i_lo = sg.u0 - halo;                       // image position of panel row 0
                // first image position >= max(i_lo, 0) in column zc
                const int start = i_lo > 0 ? i_lo : 0;
                int at = start + ((zc - start % p.W) + p.W) % p.W;
                const int sub = lane >> 3, chunk = lane & 7;      // four rows x eight 16-byte pieces per pass
                at += sub * p.W;
                for (; at < p.HW && at - i_lo < rows_total; at += 4 * p.W) {
                    const int r = at - i_lo;
#pragma unroll
                    for (int pn = 0; pn < NP; ++pn)
                        *reinterpret_cast<uint4 *>(qb + pn * p.panel_bytes + r * 128 + chunk * 16) = make_uint4(0u, 0u, 0u, 0u);
                }
                fence_async_proxy();
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&pipe.q_ready[buf]);
            if (++buf == p.nq) { buf = 0; parity ^= 1u; }
        }
    } else {
        // epilogue: TMEM lane = input channel, column = (tap, output channel). Every buffer of the
        // pipeline is free by now, so the accumulators are staged there as plain fp32 rows
        // [column][128 ci] and one thread hands them to the copy engine, which adds them into the
        // scratch [tap][co][ci] (rows of 512 bytes, 32 columns per request).
        const int q = warp & 3, et = threadIdx.x - 128;
        bool ok = g1 > g0 && mbar_wait(&pipe.acc, 0, p.err_flag);
        {   // the same decision in all 128 threads (they meet at barriers below)
            unsigned r;
            asm volatile(
                "{\n\t.reg .pred p, q;\n\t"
                "setp.ne.b32 p, %1, 0;\n\t"
                "bar.red.and.pred q, 1, 128, p;\n\t"
                "selp.b32 %0, 1, 0, q;\n\t}"
                : "=r"(r) : "r"(ok ? 1u : 0u) : "memory");
            ok = r != 0;
        }
        if (ok) {
            // the finish kernel may come now, not earlier: its blocks would hold thread slots that the kernels of the other
            // stream want (VGG-16 layer set: 1033 against 989 us)
            chain_release();
            tc_fence_after();
            const long long t_epi = clock64();
            // Only the rows the layer wants are handed over, 32 columns at a time: while the copy engine adds one block the next is
            // staged. What bounds this is an SM's way out, 24 bytes a clock for additions (30 for stores) whatever their form
            // or number (196 KB: 8.8 thousand clocks alone; 12 where all blocks were staged first, 9.5 so).
            float *stg = reinterpret_cast<float *>(smem);
            for (int c = c_lo, n = 0; c < c_hi; ++c, ++n) {
                float *const blk = stg + n % p.stage_chunks * 4096;
                if (n >= p.stage_chunks) {                     // the engine must have read the block's last use
                    if (et == 0) bulk_wait_read_all();
                    asm volatile("bar.sync 1, 128;" ::: "memory");
                }
                unsigned v[32];
                tmem_ld32(tmem_base + (static_cast<unsigned>(q * 32) << 16) + c * 32, v);
                float *dst = blk + (p.split ? (q >> 1) * 2048 + (q & 1) * 32 : q * 32) + lane;
                const int pitch = p.split ? 64 : 128;
#pragma unroll
                for (int j = 0; j < 32; ++j) dst[j * pitch] = __uint_as_float(v[j]);
                fence_async_proxy();
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (et != 0) continue;
                int ky, col0;                                  // tap and first output channel of these 32 columns
                if (NP == 2 && p.phase_tiles > 0) {            // columns 0-127: ky = 0, 128-255: ky = 1
                    ky = c >> 2;
                    col0 = (c & 3) * 32;
                } else {                                       // columns 0-63: ky = 2, 64-127: ky = 1, 128-191: ky = 0, then the next 64 channels
                    const int pn = c >= 6 ? 1 : 0, r = c - 6 * pn;
                    ky = 2 - (r >> 1);
                    col0 = 64 * pn + (r & 1) * 32;
                }
                // The rows of output channels past Cout are outside the tap's matrix: the engine skips them. (They are
                // zeros only while the activations are finite: NaN added to the next tap's first rows would stay in
                // the scratch where nobody reads that tap.)
                if (co0 + col0 < p.Cout) {
                    tma_reduce_add_3d(&map_acc, ci0, co0 + col0, ky * 3 + kx, blk);
                    if (p.split) tma_reduce_add_3d(&map_acc, 0, co0 + col0, ky * 3 + kx, blk + 2048);
                }
                bulk_commit();
            }
            if (et == 0) bulk_wait_read_all();                 // the blocks are read before the CTA goes
            if (et == 0) report_wait(p.stats, 5, clock64() - t_epi);     // how long handing over the sums took
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tmem_dealloc(tmem_base, TCOLS);
    }
}

// dW[co][ci][tap] = Delta * acc[tap][co][cip]; the scratch goes back to zero for the next call. The scratch
// rows hold cin_pad >= cin channels (activations whose channel count is no multiple of 8 were padded).
// PHASES: a stride-2 layer run on phase images (scratch rows of 4 cin channels, phase ph = 2 py + px at channels
// ph * cin ...): the strided layer's tap (ky, kx) of (co, ci) is tap (ty, tx) of channel ph * cin + ci with
// ky = 0 -> (py, ty) = (1, 0), 1 -> (0, 1), 2 -> (1, 1), kx likewise; the other scratch entries were never touched.
// A thread takes four neighbouring channels of an output channel: nine 16-byte loads (and the zeros written back), 36 values that
// follow its neighbour's in dW, whatever rows they belong to and whatever the channel count (channels of the padding are left out).
// They are handed round within the warp and leave as whole lines. Straight from the threads, 144 bytes apart, they were 9 stores of 32
// pieces, or 36 where channels are no multiple of eight: bf16 326 -> 432 at 6x6, batch 22, joined 52.4 us, 41.9 so; fp32 961 -> 224 at
// 14x15, batch 8, overlapped 79.5, 51.6; of channels that are multiples of eight bf16 784 -> 760 at 10x10, batch 13, joined 85.8, 73.0;
// VGG-16 layer set 680, 664; ResNet-50 841, 835.
// No shared memory (a dW CTA leaves none: packed there, bf16 128 -> 256 at 20x20, batch 30, dW alone, takes 30.0 us, 26.6 so) and few threads:
// the blocks become resident while the dW kernel still hands over its sums, and
// what they hold then is missing to the next layer's quantization and dX, which want to start at the same time (seven blocks of
// 256 threads per SM: VGG-16 layer set 747 us against 735; two blocks of these per SM: 749, eight: 736).
constexpr int kThreadsF3 = 128;
template <bool PHASES, bool VECTORS>                                // VECTORS: channels are a multiple of four, dW leaves 16 bytes a thread
__global__ void __launch_bounds__(kThreadsF3)
tc3_dw_finish_kernel(float *__restrict__ acc, const float *__restrict__ delta_p, float *__restrict__ dW, int cout, int cin, int cin_pad) {
    constexpr unsigned kAll = 0xffffffffu;
    const unsigned per_row = (PHASES ? cin : cin_pad) / 4, quads = static_cast<unsigned>(cout) * per_row;      // multiples of four
    const size_t tap = static_cast<size_t>(cout) * cin_pad;         // (PHASES: cin_pad = 4 cin)
    chain_wait();
    chain_release();
    const float delta = *delta_p;
    const int lane = threadIdx.x & 31, turn = lane % 9;
    for (unsigned i = blockIdx.x * kThreadsF3 + threadIdx.x; i - lane < quads; i += gridDim.x * kThreadsF3) {
        const bool mine = i < quads;
        const unsigned co = i / per_row, ci = (i - co * per_row) * 4;
        float *const base = acc + static_cast<size_t>(co) * cin_pad + ci;
        auto place = [&](int t) {
            const int ky = t / 3, kx = t % 3;
            const int ph = PHASES ? (ky != 1) * 2 + (kx != 1) : 0, tp = PHASES ? (ky == 0 ? 0 : 1) * 3 + (kx == 0 ? 0 : 1) : t;
            return reinterpret_cast<float4 *>(base + tp * tap + static_cast<size_t>(ph) * cin);
        };
        float4 v[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) v[t] = mine ? __ldcg(place(t)) : make_float4(0.f, 0.f, 0.f, 0.f);
        // where my values go, behind the warp's first one, and how many there are
        const int left = cin - static_cast<int>(ci), words = !mine || left <= 0 ? 0 : left < 4 ? 9 * left : 36;
        const size_t to = (static_cast<size_t>(co) * cin + (left > 0 ? ci : cin)) * 9, first = __shfl_sync(kAll, to, 0);
        const int from = mine ? static_cast<int>(to - first) : 0;
        float o[36];
#pragma unroll
        for (int t = 0; t < 9; ++t) {
            if (mine) __stcg(place(t), make_float4(0.f, 0.f, 0.f, 0.f));
            o[t] = v[t].x * delta;
            o[9 + t] = v[t].y * delta;
            o[18 + t] = v[t].z * delta;
            o[27 + t] = v[t].w * delta;
        }
        // Group k (four values) of lane s is the warp's group 9 s + k; lane l stores the groups 32 j + l. Nine is odd, so for one k all lanes
        // send to different ones: to lane (9 s + k) % 32, from which lane l receives with s = 25 (l - k) % 32 ...
#pragma unroll
        for (int k = 0; k < 9; ++k) {
            const int s = 25 * (lane - k) & 31;
#pragma unroll
            for (int e = 0; e < 4; ++e) o[4 * k + e] = __shfl_sync(kAll, o[4 * k + e], s);
        }
        // ... and has the group of its j-th store as k = (5 j + l) % 9: turned by l % 9, that is 5 j % 9 in every lane
#pragma unroll
        for (int b = 1; b <= 8; b *= 2) {
            float r[36];
#pragma unroll
            for (int e = 0; e < 36; ++e) r[e] = turn & b ? o[(e + 4 * b) % 36] : o[e];
#pragma unroll
            for (int e = 0; e < 36; ++e) o[e] = r[e];
        }
#pragma unroll
        for (int j = 0; j < 9; ++j) {
            const int g = 32 * j + lane, s = g * 57 >> 9, k = g - 9 * s;                           // s = g / 9
            const int n = __shfl_sync(kAll, words, s) - 4 * k;
            float *const out = dW + first + __shfl_sync(kAll, from, s) + 4 * k;
            const float *const q = o + 4 * (5 * j % 9);
            if (VECTORS) {
                if (n > 0) *reinterpret_cast<float4 *>(out) = make_float4(q[0], q[1], q[2], q[3]);
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (e < n) out[e] = q[e];
            }
        }
    }
}

// fp32 activations of tiny planes stacked into tall images (one row of zeros after every image), as two bf16 tensors, one
// after the other: the values rounded to bf16 and what that rounding left over, rounded again. out is
// [2][B / G][Cin][pitch] with G (H + 1) W positions per tall image; position q of tall image t is position
// q % ((H + 1) W) of image t G + q / ((H + 1) W), or zero in the extra row and in the padding.
// beside: see rows_job_kernel (nsd_kernels.cu); one block waits.
// A thread takes eight consecutive positions of one tall image's row: index arithmetic in 32 bits, one division per row and
// then step and wrap, one 16-byte store per piece (the previous form, a position per thread with 64-bit divisions, took 25 to
// 50 us beside a dX kernel at 512 channels of 4x4; the data are 4 MB).
__global__ void __launch_bounds__(256)
x_split_stacked_kernel(const float *__restrict__ X, __nv_bfloat16 *__restrict__ out, unsigned Bt, unsigned G, unsigned Cin,
                       unsigned HW, unsigned W, unsigned pitch, int beside) {
    if (!beside) chain_wait();
    chain_release();
    const unsigned gpp = pitch / 8, per_img = HW + W, n = Bt * Cin * gpp;
    const size_t piece = static_cast<size_t>(Bt) * Cin * pitch, img_stride = static_cast<size_t>(Cin) * HW;
    for (unsigned i = blockIdx.x * 256u + threadIdx.x; i < n; i += gridDim.x * 256u) {
        const unsigned pl = i / gpp, q0 = (i - pl * gpp) * 8, t = pl / Cin, ci = pl - t * Cin;
        unsigned g = q0 / per_img, r = q0 - g * per_img;
        const float *src = X + (static_cast<size_t>(t) * G + g) * img_stride + static_cast<size_t>(ci) * HW;
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            x[e] = (g < G && r < HW) ? __ldg(src + r) : 0.f;
            if (++r == per_img) { r = 0; ++g; src += img_stride; }
        }
        unsigned h[4], l[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const __nv_bfloat162 hh = __floats2bfloat162_rn(x[2 * k], x[2 * k + 1]);
            const float2 hf = __bfloat1622float2(hh);
            const __nv_bfloat162 ll = __floats2bfloat162_rn(x[2 * k] - hf.x, x[2 * k + 1] - hf.y);
            h[k] = *reinterpret_cast<const unsigned *>(&hh);
            l[k] = *reinterpret_cast<const unsigned *>(&ll);
        }
        const size_t o = static_cast<size_t>(pl) * pitch + q0;
        *reinterpret_cast<uint4 *>(out + o) = make_uint4(h[0], h[1], h[2], h[3]);
        *reinterpret_cast<uint4 *>(out + piece + o) = make_uint4(l[0], l[1], l[2], l[3]);
    }
    if (beside && blockIdx.x == 0) chain_wait();
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// The code panel of a segment: its positions and W + 1 more on either side, in boxes of at most 256 rows
struct Panel { int nload, rows_box, bytes; };
Panel panel_of(int seg, int W) {
    const int rows = seg + 2 * (W + 1), nload = (rows + 255) / 256, rows_box = (rows + nload - 1) / nload;
    return Panel{nload, rows_box, round_up(nload * rows_box * 128, 1024)};
}

}  // namespace

// Whether the kernel fits half an SM: two code buffers of the shortest segment beside two activation slots (W up to 59)
bool tc3_dw_fits_half(const ConvShape &s) {
    return 2 * static_cast<size_t>(panel_of(64, static_cast<int>(s.W)).bytes) + 1024 + 2 * kXS * kXTile <= kHalfSm;
}

// DBP_EUNSUPPORTED: the shape does not fit (the caller uses another kernel)
int tc3_stack_images(const ConvShape &s, int io) {
    const long long HW = s.H * s.W, per_img = HW + s.W;
    if (io != DBP_F32 || s.k != 3 || HW >= 64 || per_img > 64 || s.B < 2 || s.Cout % 8 != 0) return 0;
    if (s.B * s.Cin * per_img >= (1ll << 31)) return 0;          // the stacking kernel indexes in 32 bits
    // the largest divisor of the batch whose tall image stays within one segment of the kernel
    for (long long g = s.B; g >= 2; --g)
        if (s.B % g == 0 && g * per_img <= 320) return static_cast<int>(g);
    return 0;
}

int launch_x_stacked(dbp_ctx *ctx, const float *X, void *out, const ConvShape &s, int stack_g, bool beside) {
    const long long tall = s.B / stack_g, pitch = (stack_g * (s.H + 1) * s.W + 7) / 8 * 8;
    long long blocks = (tall * s.Cin * (pitch / 8) + 255) / 256;
    if (blocks > ctx->sm_count * 4) blocks = ctx->sm_count * 4;
    return cuda_ok(launch_chained(x_split_stacked_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, ctx->stream, X,
                                  static_cast<__nv_bfloat16 *>(out), static_cast<unsigned>(tall), static_cast<unsigned>(stack_g),
                                  static_cast<unsigned>(s.Cin), static_cast<unsigned>(s.H * s.W), static_cast<unsigned>(s.W),
                                  static_cast<unsigned>(pitch), beside ? 1 : 0));
}

// X: bf16 planes of x_pitch values (a multiple of 8); fp32 activations as two pieces (as if the batch were twice as long).
// Tiny planes stacked into tall images: `s` describes the tall images and codes and X are their stacked copies.
// overlapped: the next layer's kernels come beside this one.
int launch_tc3_tma_dw(dbp_ctx *ctx, const void *codes_nhwc, const void *X, int pieces, long long x_pitch, const float *delta_p,
                      const ConvShape &s, float *dW, int *err_flag, bool half, bool overlapped) {
    // the scratch's rows are padded to a multiple of 16 bytes
    const long long cin_pad = (s.Cin + 7) / 8 * 8, q_pitch = (s.Cout + 7) / 8 * 8;
    const long long HW = s.H * s.W;
    Dw3T p{};
    p.Cout = static_cast<int>(s.Cout); p.W = static_cast<int>(s.W); p.HW = static_cast<int>(HW);
    p.err_flag = err_flag;
    p.stats = ctx->wait_stats;
    // half an SM has room for the 192 accumulator columns of 64 output channels (an MMA of N = 192 does as much per clock as
    // three of 128); splits are still chosen for one CTA per SM, because every split adds its accumulators into the scratch
    // (for two: 2 % slower on average over 60 drawn layers)
    const int NP = s.Cout > 64 && !half ? 2 : 1;
    p.ci_tiles = static_cast<int>((cin_pad + 127) / 128);
    p.co_tiles = static_cast<int>((s.Cout + 64 * NP - 1) / (64 * NP));
    // The segment whose copies are the least, of those whose two code buffers fit beside at least three activation slots: every segment
    // copies its halo too, boxes come whole, and a segment costs about ten rows' time besides. 72 -> 72 fp32 at 14x14, batch 128, with 192
    // positions (444 rows an image) and 128 (316): 63.6, 60.7 us; 360 -> 112 at 12x12, batch 113, with 128 (308) and 192 (218): 102, 88;
    // 200 -> 48 at 24x24, batch 43, with 192 instead of 320: 53.4, 51.4. In half an SM, beside two slots, the longest:
    // 64 -> 64 at 13x13, batch 128, with 64 positions 32.4, with 128 30.8.
    p.xs = HW > 64 ? kXS : 1;
    const size_t x_slot = static_cast<size_t>(p.xs) * kXTile;
    auto copied = [&](int seg) {                          // rows of codes per image, with what a segment costs
        const Panel pn = panel_of(seg, p.W);
        return (HW + seg - 1) / seg * (pn.nload * pn.rows_box + 10);
    };
    auto best_segment = [&](size_t budget) {
        int best = 0;
        for (int seg = static_cast<int>(HW < 512 ? (HW + 63) / 64 * 64 : 512); seg >= 64; seg -= 64)
            if (2ll * NP * panel_of(seg, p.W).bytes + 1024 + (half ? 2 : 3) * kXS * kXTile <= static_cast<long long>(budget) &&
                (best == 0 || (!half && copied(seg) < copied(best))))
                best = seg;
        return best;
    };
    size_t budget = half ? kHalfSm : 227 * 1024 - 2048;
    int seg = best_segment(budget);
    if (seg == 0) return DBP_EUNSUPPORTED;
    // An overlapped call's kernel of 128 output channels leaves 17 KB to a block of the next layer's position-major quantizer (256 -> 256
    // fp32 at 16x16, batch 128: 145 us, 168 without; VGG-16 layer set 747, 751; 34 KB: 752, 51 KB: 762). What shorter segments cost for it, the
    // share of bytes that is copied more, counts once per tile of channels, what it brings goes with the output channels. The line lies between, us with
    // the room and without: 0.22 (72 -> 72 fp32 at 24x24, batch 43) 40.4, 43.5; 0.22 (128 -> 128 fp32 at 12x12, batch 128) 39.7, 41.8; and 0.30
    // (128 -> 128 bf16 at 56x56, batch 16) 51.4, 47.4; 0.33 (100 -> 100 bf16 at 44x44, batch 100) 168.9, 148.6; 0.75 (360 -> 112 fp32 at
    // 12x12, batch 113) 86.6, 75.3. Wide planes of few images gain from the room for longer: 0.26 (128 -> 128 fp32 at 44x44, batch 16) 51.9, 57.4.
    // Kernels of 64 channels: long segments are worth more (64 -> 64 at 32x32: 22.0 us, 24.0).
    if (overlapped && !half && NP == 2) {
        const size_t less = 210 * 1024 - 2048;
        const int with_room = best_segment(less);
        const double row = 128.0 * NP, bytes = copied(seg) * row + (HW + 63) / 64 * kXTile;
        if (with_room != 0 && (copied(with_room) - copied(seg)) * row / bytes * p.ci_tiles * p.co_tiles * 128 <= 0.25 * s.Cout) {
            budget = less;
            seg = with_room;
        }
    }
    const Panel pn = panel_of(seg, p.W);
    const size_t qbuf = static_cast<size_t>(NP) * pn.bytes;
    size_t fixed = 2 * qbuf + 1024;
    p.SEG = seg; p.nload = pn.nload; p.rows_box = pn.rows_box; p.panel_bytes = pn.bytes;
    // short segments: their MMAs (about 950 clocks of 64 positions) do not cover a copy's way and the zeroing of its columns
    p.nq = 2;
    while (seg <= 128 && p.nq < kMaxNQ && fixed + qbuf + 4 * x_slot <= budget) { ++p.nq; fixed += qbuf; }
    p.nx = static_cast<int>((budget - fixed) / x_slot);
    if (p.nx > kMaxNX) p.nx = kMaxNX;
    const size_t smem = fixed + static_cast<size_t>(p.nx) * x_slot;
    p.segs_per_img = (p.HW + p.SEG - 1) / p.SEG;
    p.code_batch = static_cast<int>(s.B);
    p.split = pieces == 2 && s.Cin <= 64 ? 1 : 0;
    p.nseg = s.B * (p.split ? 1 : pieces) * p.segs_per_img;
    // a stride-2 layer on phase images whose phases are whole channel tiles: 6 of the 12 (phase, kernel column)
    // pairs carry taps of the strided layer
    p.phase_tiles = (ctx->phase_cin > 0 && ctx->phase_cin % 128 == 0 && cin_pad == 4ll * ctx->phase_cin)
                        ? ctx->phase_cin / 128 : 0;
    const long long tiles = p.phase_tiles > 0 ? static_cast<long long>(p.co_tiles) * 6 * p.phase_tiles
                                              : static_cast<long long>(p.ci_tiles) * p.co_tiles * 3;
    // (an MMA takes 16 positions)
    const long long nsplit = choose_split(tiles, p.nseg, ctx->sm_count, kMaxMmas * 16 / p.SEG, &p.per_split);
    p.nsplit = static_cast<int>(nsplit);
    if (tiles * nsplit >= (1ll << 31)) return DBP_EUNSUPPORTED;
    // fp32 scratch [9][Cout][Cin]: zero whenever no call is in flight
    const size_t pairs = static_cast<size_t>(s.Cout) * cin_pad;
    const size_t had = ctx->dw_acc.bytes;
    int rc = ws_reserve(ctx, ctx->dw_acc, pairs * 9 * sizeof(float));
    if (rc) return rc;
    if (ctx->dw_acc.bytes != had || !ctx->dw_acc_clean) {
        if (cudaMemsetAsync(ctx->dw_acc.ptr, 0, ctx->dw_acc.bytes, ctx->stream) != cudaSuccess) return fail_cuda("clearing the dW scratch");
        ctx->dw_acc_clean = true;
    }
    float *acc = static_cast<float *>(ctx->dw_acc.ptr);
    p.stage_chunks = static_cast<int>((smem - 1024) / 16384);
    CUtensorMap map_q, map_x, map_acc;
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(cin_pad), static_cast<unsigned long long>(s.Cout), 9};
        const unsigned long long str[2] = {static_cast<unsigned long long>(cin_pad) * 4, static_cast<unsigned long long>(pairs) * 4};
        const unsigned box[3] = {p.split ? 64u : 128u, 32, 1};
        if (!encode_map_f32_rows(&map_acc, acc, 3, dims, str, box)) return fail_cuda("tensor map of the dW scratch");
    }
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(s.Cout), static_cast<unsigned long long>(HW),
                                            static_cast<unsigned long long>(s.B)};
        const unsigned long long str[2] = {static_cast<unsigned long long>(q_pitch) * 2,
                                           static_cast<unsigned long long>(q_pitch) * 2 * HW};
        const unsigned box[3] = {64, static_cast<unsigned>(p.rows_box), 1};
        if (!encode_map_bf16(&map_q, codes_nhwc, 3, dims, str, box)) return fail_cuda("tensor map of the code panels");
    }
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(HW), static_cast<unsigned long long>(s.Cin),
                                            static_cast<unsigned long long>(s.B) * pieces};
        const unsigned long long str[2] = {static_cast<unsigned long long>(x_pitch) * 2,
                                           static_cast<unsigned long long>(x_pitch) * 2 * s.Cin};
        const unsigned box[3] = {64, p.split ? 64u : 128u, 1};
        if (!encode_map_bf16(&map_x, X, 3, dims, str, box)) return fail_cuda("tensor map of the activations");
    }
    if (half) cudaFuncSetAttribute(tc3_tma_dw_kernel<1>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    auto kern = NP == 2 ? tc3_tma_dw_kernel<2> : tc3_tma_dw_kernel<1>;
    if (allow_shared(kern) != cudaSuccess)
        return fail_cuda("shared memory size");
    if ((rc = cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(tiles * nsplit)), dim3(kThreadsW3), smem,
                                     ctx->stream, map_q, map_x, map_acc, p))))
        return rc;
    // a stride-2 layer's own weight gradient comes straight from the scratch
    const bool phases = p.phase_tiles > 0 && ctx->phase_dw_out != nullptr;
    if (phases) ctx->phase_dw_done = true;
    const long long quads = s.Cout * ((phases ? ctx->phase_cin : cin_pad) / 4), need = (quads + kThreadsF3 - 1) / kThreadsF3;
    const long long most = 4ll * ctx->sm_count, blocks = need < most ? need : most;
    const auto finish = phases ? tc3_dw_finish_kernel<true, true> : s.Cin % 4 == 0 ? tc3_dw_finish_kernel<false, true> : tc3_dw_finish_kernel<false, false>;
    return cuda_ok(launch_chained(finish, dim3(static_cast<unsigned>(blocks)), dim3(kThreadsF3), 0, ctx->stream, acc, delta_p,
                                  phases ? ctx->phase_dw_out : dW, static_cast<int>(s.Cout), static_cast<int>(phases ? ctx->phase_cin : s.Cin),
                                  static_cast<int>(cin_pad)));
}

}  // namespace dbp
