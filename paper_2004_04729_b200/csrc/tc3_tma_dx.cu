// Input gradient of 3x3 convolutions (stride 1, pad 1) on the tensor cores, both operands brought
// in by tiled copies (Eq. (qda), "analogous for convolutional layers"):
//   dX[b][ci][y][x] = Delta * sum_(co,ky,kx) q[b][co][y+1-ky][x+1-kx] * W[co][ci][ky][kx]
//
// The quantizer has written the codes position-major, [b][y][x][co] in bf16, so a patch of
// (Ht+2) x Wp positions x 64 output channels is ONE 4-D tiled copy whose out-of-image rows and
// columns the copy engine fills with zeros: the convolution's zero padding costs nothing. In
// shared memory the patch is a K-major operand, one 128-byte row of 64 channels per position,
// rows numbered r = yy * Wp + xx, xx = 0 being column -1. The output position (y, x) of the patch is
// accumulator column n = (y-y0) * Wp + x, and the code a tap (ky, kx) needs for it sits in row
// n + (2-ky) * Wp + (2-kx): a tap is only a different start row of the same operand (the 128-byte
// swizzle is a function of the shared-memory address, so a descriptor may start at any row). The
// columns that belong to the halo are computed and thrown away, so halos are shared: Wp = W + 1 (the zero
// right of a row is the zero left of the next one; bf16 rows of even W keep W + 2, which keeps pairs of
// outputs on even columns), and small images, taken several at a time along the same row space, have
// one row of zeros between them. What a tap reads behind the last row is zeroed once.
//
//   A = weights of one tap [64 co][128 ci]  (M = input channels, MN-major; from W re-laid as [tap][co][ci])
//   B = code patch         [rows][64 co]    (N = up to 256 patch positions, K-major)
//   K = (64-channel block of co) x (nine taps), four MMAs of 16 channels each; for fp32 weights (two bf16 pieces)
//       both pieces of a block, or, in long reductions, the low pieces of all blocks before the high ones
//
// An MMA of N columns takes max(N/2, 32 + N/4) clocks (measured; the second term is its operands' way out of shared
// memory: 4 KB of A, 32 bytes per column of B), and streamed weights take shared-memory and L2 bandwidth on top. So N is
// made large, and where that leaves fewer tiles than SMs the reduction over co is split over a cluster of KS CTAs, whose
// partial sums are read through distributed shared memory and added in rank order (fixed: dX does not depend on timing).
// fp32 layers of at most 64 input channels put the two pieces of their weights on the two halves of the accumulator's
// lanes (9 taps instead of 18 with half-empty MMAs); the halves are added on the way out.
//
// A CTA is persistent over (patch, 128-channel block of ci) tiles. Warp 0 copies code patches,
// warp 1 copies weight tiles, warps 2 and 3 issue the MMAs of alternate tiles into two accumulators in tensor
// memory, warps 4-19 drain them: scale by Delta, convert, compact the valid columns into a
// shared staging block [ci][positions] and write whole runs of consecutive positions per channel.
// Every wait is bounded.
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace tc;

template <bool LEAN>
constexpr int kEpiWarps = LEAN ? 8 : 16;
template <bool LEAN>
constexpr int kThreads3 = (4 + kEpiWarps<LEAN>) * 32;            // copy, copy, MMA, MMA, epilogue warps
constexpr int kWPanel = 8192;                    // [64 co][64 ci] bf16
constexpr int kMaxQ = 2;                         // code patches in flight
constexpr int kMaxW = 18;                        // weight slots (ring, or all of them when they stay resident)
constexpr int kAccCols = 256;
constexpr int kBlock = 32 * 128;                 // one epilogue warp's [32 ci][128 bytes of positions], swizzled

struct Dx3T {
    const float *delta_p;
    void *dX;
    int B, Cin, Cout, H, W, Wp;
    int KS;                       // CTAs (a cluster) that share a tile's reduction; > 1: one tile per cluster
    int split;                    // the low piece of the weights is the upper panel (fp32, Cin <= 64)
    int slots;                    // weight slots per block of co and pass (in phase mode of the tiles with one live kernel row)
    int passes;                   // 2: the low pieces of the weights first, over all blocks of co, then the high ones
    int Ht;                       // image rows per patch
    int nb;                       // images per patch (> 1 only when Ht == H)
    int tiles_y;                  // patches per image (nb == 1)
    int img_rows;                 // patch rows per image: (Ht + 2) * Wp, or (H + 1) * Wp with several images
    int N;                        // accumulator columns in use (multiple of 16)
    int q_bytes;                  // bytes of one patch buffer (multiple of 1024)
    int q_tx;                     // bytes one patch copy delivers
    int ncb;                      // 64-channel blocks of co
    int ci_tiles;
    long long pos_tiles, ntiles;
    int a_panels;                 // 64-channel panels of ci per weight tile (1 or 2)
    int ntaps;                    // 9, or 18 for fp32 weights split into two bf16 pieces (taps 9-17: the low pieces)
    int es;                       // bytes per element of dX (2 or 4)
    int G;                        // taps per weight slot (one hand-over): 9, 3 or 1; phase mode: 2
    int w_slot;                   // bytes of a weight slot, [panel][tap][64 co][64 ci]: a_panels * G * 8 KB
    int nq, nw;                   // ring sizes
    int resident;                 // the weights of all taps and co blocks stay in shared memory (one ci block)
    int run;                      // Ht * W: staged positions per image
    int off_at;                   // where the column table lies
    int pitch;                    // bytes per channel row of the staging block (an odd number of words)
    int pairs;                    // W even: columns are staged two at a time
    int unit;                     // > 0: blocks of 32 channels x 128 bytes of consecutive positions leave by the copy engine;
                                  // the largest power of two up to 32 that divides W
    unsigned w_rcp;               // ceil(2^16 / W): i / W = i w_rcp >> 16 for i < 512, W <= 62
    int phase_cin;                // > 0: the layer is a stride-2 layer on phase images (channel block ph * phase_cin ...
                                  // holds phase ph = 2 py + px); a phase's weights are zero outside the taps
                                  // ky in {1} (py = 0) or {0, 1} (py = 1), kx likewise, and those taps are skipped
    int *err_flag;
    unsigned long long *stats;    // wait counters (may be null)
};

struct PipeX {
    unsigned long long q_full[kMaxQ], q_empty[kMaxQ], w_full[kMaxW], w_empty[kMaxW], acc_full[2], acc_empty[2], turn[2];
    unsigned tmem_base;
};

__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1, int c2, int c3,
                                            unsigned long long *bar) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(map), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, int c0, int c1, int c2, int c3, const void *src) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%2, %3, %4, %5}], [%1];"
                 ::"l"(map), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}

// U accumulator columns (the caller waits)
template <int U>
__device__ __forceinline__ void tmem_ld_cols(unsigned taddr, unsigned *r) {
    if constexpr (U == 4) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr));
    } else if constexpr (U == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr));
    } else {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                       "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr));
    }
}
// the accumulators of 32 consecutive positions from position i0 of an image's part of the patch on (rows of W positions lie Wp
// columns apart, and U divides W); positions from `limit` on, which nobody stores, read some column that exists
template <int U>
__device__ __forceinline__ void load_positions(unsigned base, int i0, int limit, const Dx3T &p, unsigned (&v)[32]) {
#pragma unroll
    for (int k = 0; k < 32; k += U) {
        const int i = i0 + k, y = static_cast<int>(static_cast<unsigned>(i) * p.w_rcp >> 16);
        tmem_ld_cols<U>(base + (i < limit ? i + y * (p.Wp - p.W) : 0), v + k);
    }
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void load_positions(unsigned base, int i0, int limit, const Dx3T &p, unsigned (&v)[32]) {
    if (p.unit >= 16) load_positions<16>(base, i0, limit, p, v);
    else if (p.unit == 8) load_positions<8>(base, i0, limit, p, v);
    else load_positions<4>(base, i0, limit, p, v);
}

// dst[0 .. n) = value(0 .. n), lanes along the run, four values per lane in flight
template <typename T, typename F>
__device__ __forceinline__ void copy_run(T *dst, int n, int lane, const F &value) {
    for (int i0 = lane; i0 < n; i0 += 128) {
        T v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + 32 * u < n) v[u] = value(i0 + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (i0 + 32 * u < n) dst[i0 + 32 * u] = v[u];
    }
}

// All threads of the cluster; writes to distributed shared memory before it are visible behind it.
__device__ __forceinline__ void cluster_barrier() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Barrier over the epilogue threads that also tells every one of them whether all of them are
// still fine: a thread whose bounded wait ran out arrives like the others, so nobody is left waiting.
template <int THREADS>
__device__ __forceinline__ bool epilogue_all(bool mine) {
    unsigned r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.b32 p, %1, 0;\n\t"
        "bar.red.and.pred q, 1, %2, p;\n\t"
        "selp.b32 %0, 1, 0, q;\n\t}"
        : "=r"(r) : "r"(mine ? 1u : 0u), "n"(THREADS) : "memory");
    return r != 0;
}

// BLOCKS: dX leaves in blocks by the copy engine (p.unit > 0, p.KS == 1); an instance of its own because the other paths' code
// in the same kernel costs each of them 3 %
// LEAN: half an SM (shared memory, tensor memory, registers): one tile per CTA, a dW CTA beside it
template <bool BLOCKS, bool LEAN>
__global__ void __launch_bounds__(kThreads3<LEAN>, LEAN ? 2 : 1)
tc3_tma_dx_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_w,
                  const __grid_constant__ CUtensorMap map_o, const __grid_constant__ CUtensorMap map_t, const Dx3T p) {
    constexpr int kThreadsX = kThreads3<LEAN>, EW = kEpiWarps<LEAN>, kEpiThreads = EW * 32, PARTS = EW / 4;
    constexpr unsigned kTmem = LEAN ? kAccCols : 2 * kAccCols;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    unsigned char *q_s = smem;                                   // nq code patches
    unsigned char *w_s = q_s + p.nq * p.q_bytes;                 // nw weight slots
    // one tile per CTA: the staging block lies over the operands, which nobody reads any more by then
    unsigned char *stage = LEAN ? smem : w_s + p.nw * p.w_slot;  // [128 ci][pitch], or a 4 KB block per epilogue warp
    short *s_off = reinterpret_cast<short *>(LEAN ? smem + p.off_at : stage + (BLOCKS ? EW * kBlock : 128 * p.pitch));   // column -> staged position (or -1), 256 entries
    __shared__ PipeX pipe;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KS = BLOCKS ? 1 : p.KS;
    const int rank = KS > 1 ? static_cast<int>(blockIdx.x) % KS : 0;      // consecutive CTAs are a cluster
    const long long t_first = blockIdx.x / KS, t_step = gridDim.x / KS;
    const int c_lo = rank * p.ncb / KS, c_hi = (rank + 1) * p.ncb / KS;   // my 64-channel blocks of co

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxQ; ++s) { mbar_init(&pipe.q_full[s], 1); mbar_init(&pipe.q_empty[s], 1); }
        for (int s = 0; s < kMaxW; ++s) { mbar_init(&pipe.w_full[s], 1); mbar_init(&pipe.w_empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&pipe.turn[a], 1); mbar_init(&pipe.acc_full[a], 1); mbar_init(&pipe.acc_empty[a], kEpiThreads / 32); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_w);
        if (BLOCKS) { tma_prefetch_desc(&map_o); tma_prefetch_desc(&map_t); }
    }
    if (warp == 2) tmem_alloc(&pipe.tmem_base, kTmem);
    // which accumulator columns hold an output, and where it goes in a channel's staged run
    if (threadIdx.x >= 128 && threadIdx.x < 384) {
        const int n = threadIdx.x - 128;
        const int img = n / p.img_rows, rem = n - img * p.img_rows;
        const int yy = rem / p.Wp, xx = rem - yy * p.Wp;
        s_off[n] = (n < p.N && img < p.nb && yy < p.Ht && xx < p.W) ? static_cast<short>(img * p.run + yy * p.W + xx) : static_cast<short>(-1);
    }
    // the rows behind a patch: the last row's right-hand zero and the zeros below the last image; copies never reach them
    for (int q = 0; q < p.nq; ++q)
        for (int i = p.img_rows * p.nb * 8 + threadIdx.x; i < p.q_bytes / 16; i += kThreadsX)
            reinterpret_cast<uint4 *>(q_s + q * p.q_bytes)[i] = make_uint4(0u, 0u, 0u, 0u);
    fence_async_proxy();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = pipe.tmem_base;
    if (KS > 1) cluster_barrier();       // every CTA of the cluster is there before anybody writes into its staging block
    // everything above touched only this CTA's shared and tensor memory
    chain_wait();

    // tile t -> (patch, ci block); patch -> first image and first image row
    auto tile_of = [&](long long t, int &ci0, int &b0, int &y0) {
        const long long pt = t / p.ci_tiles;
        ci0 = static_cast<int>(t - pt * p.ci_tiles) * 128;
        if (p.nb == 1) {
            b0 = static_cast<int>(pt / p.tiles_y);
            y0 = static_cast<int>(pt - static_cast<long long>(b0) * p.tiles_y) * p.Ht;
        } else {
            b0 = static_cast<int>(pt) * p.nb;
            y0 = 0;
        }
    };
    // Weight slots per 64-channel block of co. In phase mode a slot is one kernel row's taps kx = 0, 1, and only rows that
    // carry weights in the tile's phase have one: ky = 1 (py = 0), or ky = 0 and 1 (py = 1).
    auto phase_of = [&](long long t) { return static_cast<int>(t % p.ci_tiles) * 128 / p.phase_cin; };
    auto slots_of = [&](long long t) { return p.phase_cin > 0 && (phase_of(t) & 2) ? 2 * p.slots : p.slots; };
    // what a tile goes through: blocks of co, in two passes once with the low and once with the high pieces of the weights
    const int ncbl = c_hi - c_lo, nblk = p.passes * ncbl;
    auto block_of = [&](int i) { return c_lo + (i < ncbl ? i : i - ncbl); };

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            unsigned parity = 1;                   // a fresh barrier passes a wait on the previous phase
            bool ok = true;
            long long waited = 0;
            for (long long t = t_first; t < p.ntiles && ok; t += t_step) {
                int ci0, b0, y0;
                tile_of(t, ci0, b0, y0);
                for (int i = 0; i < nblk; ++i) {
                    ok = mbar_wait_timed(&pipe.q_empty[s], parity, p.err_flag, waited);
                    if (!ok) break;
                    mbar_expect_tx(&pipe.q_full[s], static_cast<unsigned>(p.q_tx));
                    tma_load_4d(q_s + s * p.q_bytes, &map_q, block_of(i) * 64, -1, y0 - 1, b0, &pipe.q_full[s]);
                    if (++s == p.nq) { s = 0; parity ^= 1u; }
                }
            }
            chain_release();       // every copy is issued: the next kernel may take the slots that come free (earlier it would
                                   // hold thread slots that the dW stream's kernels want: stride-2 set 796 against 745 us)
            report_wait(p.stats, 3, waited);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int s = 0;
            unsigned parity = 1;
            bool ok = true;
            long long waited = 0;
            for (long long t = t_first; t < p.ntiles && ok; t += t_step) {
                int ci0, b0, y0;
                tile_of(t, ci0, b0, y0);
                const int slots = slots_of(t);
                for (int i = 0; i < nblk && ok; ++i) {
                    const int c = block_of(i), low = p.passes == 2 && i < ncbl ? 1 : 0;       // low: the piece of a two-pass tile
                    for (int g = 0; g < slots; ++g) {
                        if (!p.resident) {
                            ok = mbar_wait_timed(&pipe.w_empty[s], parity, p.err_flag, waited);
                            if (!ok) break;
                        }
                        // One arrival for the whole slot, one copy per panel (all taps of the slot in one box; in phase mode
                        // the live taps one by one: a quarter of the layer's weights is what there is to copy then).
                        unsigned char *dst = w_s + s * p.w_slot;
                        if (p.phase_cin == 0) {
                            mbar_expect_tx(&pipe.w_full[s], static_cast<unsigned>(p.w_slot));
                            for (int h = 0; h < p.a_panels; ++h)
                                tma_load_3d(dst + h * p.G * kWPanel, &map_w, p.split ? 0 : ci0 + 64 * h, c * 64,
                                            g * p.G + 9 * (p.split ? h : low), &pipe.w_full[s]);
                        } else {
                            const int ph = phase_of(t), ky = (ph & 2) ? g & 1 : 1, kx0 = (ph & 1) ? 0 : 1;
                            const int piece = p.passes == 2 ? low : (ph & 2) ? g >> 1 : g;
                            mbar_expect_tx(&pipe.w_full[s], static_cast<unsigned>((2 - kx0) * 2 * kWPanel));
                            for (int kx = kx0; kx < 2; ++kx)
                                for (int h = 0; h < 2; ++h)
                                    tma_load_3d(dst + (2 * h + kx) * kWPanel, &map_w, ci0 + 64 * h, c * 64, 9 * piece + ky * 3 + kx, &pipe.w_full[s]);
                        }
                        if (++s == p.nw) { s = 0; parity ^= 1u; }
                    }
                }
                if (p.resident) break;             // one ci block: every tile uses the same weights (all slots are loaded now)
            }
            report_wait(p.stats, 4, waited);
        }
    } else if (warp < 4) {
        // Two warps issue MMAs, each for every other tile (its own accumulator): what one does between tiles (waits,
        // descriptors: more than a thousand clocks) then lies beside the other's MMAs. The whole warp runs the loop (uniform
        // control flow and operands); one elected lane issues.
        const unsigned idesc = make_idesc(128, p.N, true, false);
        // Start row of tap (ky, kx) inside the patch is (2 - ky) Wp + (2 - kx), in descriptor units (16 bytes) eight times
        // that; one tap further inside a slot is kWPanel. The three taps of a kernel row are issued by one elected lane
        // from straight-line code (a loop with address stepping and an election per tap left the tensor pipe idle for long).
        constexpr unsigned a_tap = static_cast<unsigned>(kWPanel) >> 4;
        const unsigned row_step = static_cast<unsigned>(p.Wp * 8);
        const unsigned long long q_desc = make_desc(smem_u32(q_s), 16, 1024);
        // with one panel of ci (Cin <= 64) the upper 64 rows of the MMA re-read the same panel (their results are never
        // stored) instead of whatever follows the slot
        const unsigned long long w_desc = make_desc(smem_u32(w_s), p.a_panels == 2 ? p.G * kWPanel : 0, 1024);
        const unsigned q_step = static_cast<unsigned>(p.q_bytes) >> 4, w_step = static_cast<unsigned>(p.w_slot) >> 4;
        const int slot = warp - 2;
        const unsigned tmem_d = tmem_base + slot * kAccCols;
        bool ok = true;
        long long wq = 0, ww = 0, wa = 0;
        const long long born = clock64();
        int it = slot;
        unsigned n_w = slot ? nblk * slots_of(t_first) : 0;
        for (long long t = t_first + slot * t_step; t < p.ntiles && ok; t += 2 * t_step, it += 2) {
            // ring positions of this tile's first patch and weight slot (and, behind them, of this warp's next tile)
            const unsigned n_q = static_cast<unsigned>(it) * nblk;
            const int slots = slots_of(t);
            int qs = n_q % p.nq, ws = n_w % p.nw;
            unsigned qpar = (n_q / p.nq) & 1u, wpar = (n_w / p.nw) & 1u;
            if (p.resident) { ws = 0; wpar = 0; }          // completed barriers stay passable on parity 0
            n_w += nblk * (slots + slots_of(t + t_step));
            unsigned acc_on = 0u;
            const int ph = p.phase_cin > 0 ? phase_of(t) : 0;
            ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.acc_empty[slot], ((static_cast<unsigned>(it) >> 1) & 1u) ^ 1u, p.err_flag, wa));
            // The rings' barriers may be waited for one phase ahead, not more: the other warp must have seen every stage of the
            // tile before this one arrive. It says so in front of its last slot's MMAs, which is early enough.
            if (ok && it > 0)
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.turn[slot], ((static_cast<unsigned>(it - 1) >> 1)) & 1u, p.err_flag));
            if (!ok) break;
            for (int i = 0; i < nblk && ok; ++i) {
                ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.q_full[qs], qpar, p.err_flag, wq));
                if (!ok) break;
                const unsigned long long bd0 = q_desc + static_cast<unsigned>(qs) * q_step;
                int ky = 0, kx1 = 0;                       // kernel row of the next slot (G >= 3), its tap (G == 1)
                for (int g = 0; g < slots && ok; ++g) {
                    ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.w_full[ws], wpar, p.err_flag, ww));
                    if (!ok) break;
                    if (i == nblk - 1 && g == slots - 1 && elect_one()) mbar_arrive(&pipe.turn[slot ^ 1]);
                    tc_fence_after();
                    unsigned long long ad = w_desc + static_cast<unsigned>(ws) * w_step;
                    if (p.phase_cin > 0) {
                        const unsigned long long bd = bd0 + (2 - ((ph & 2) ? g & 1 : 1)) * row_step;
                        if (elect_one()) {
                            if (ph & 1) {
#pragma unroll
                                for (int k = 0; k < 4; ++k) mma_bf16(tmem_d, ad + 128 * k, bd + 16 + 2 * k, idesc, k ? 1u : acc_on);
                            }
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                mma_bf16(tmem_d, ad + a_tap + 128 * k, bd + 8 + 2 * k, idesc, (k || (ph & 1)) ? 1u : acc_on);
                        }
                        acc_on = 1u;
                    } else if (p.G == 1) {
                        const unsigned long long bd = bd0 + (2 - ky) * row_step + (2 - kx1) * 8;
                        if (elect_one()) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_bf16(tmem_d, ad + 128 * k, bd + 2 * k, idesc, k ? 1u : acc_on);
                        }
                        acc_on = 1u;
                        if (++kx1 == 3) { kx1 = 0; if (++ky == 3) ky = 0; }       // the second piece's taps start over
                    } else {
                        for (int r = 0; r < p.G; r += 3, ad += 3 * a_tap) {
                            const unsigned long long bd = bd0 + (2 - ky) * row_step;
                            if (++ky == 3) ky = 0;
                            if (elect_one()) {
#pragma unroll
                                for (int kx = 0; kx < 3; ++kx)
#pragma unroll
                                    for (int k = 0; k < 4; ++k)   // 16 co: 16 rows of A (2048 bytes), 32 bytes along a row of B
                                        mma_bf16(tmem_d, ad + kx * a_tap + 128 * k, bd + (2 - kx) * 8 + 2 * k, idesc, kx + k ? 1u : acc_on);
                            }
                            acc_on = 1u;
                        }
                    }
                    if (!p.resident && elect_one()) mma_commit(&pipe.w_empty[ws]);
                    if (++ws == p.nw) { ws = 0; wpar ^= 1u; }
                }
                if (ok && elect_one()) mma_commit(&pipe.q_empty[qs]);
                if (++qs == p.nq) { qs = 0; qpar ^= 1u; }
            }
            if (ok && elect_one()) mma_commit(&pipe.acc_full[slot]);
        }
        if (lane == 0 && it > slot) {
            report_wait(p.stats, 0, wq);
            report_wait(p.stats, 1, ww);
            report_wait(p.stats, 2, wa);
            report_wait(p.stats, 6, clock64() - born);
            report_wait(p.stats, 7, 1);
        }
    } else if (BLOCKS) {
        // epilogue where runs of positions are whole 16-byte words: every warp by itself (no barrier of all of them, no pass
        // through a staging block shared by them) moves blocks of 32 channels x 128 bytes from the accumulator to its own
        // block of shared memory, from where the copy engine takes them. Warp (q, part): lane quarter q, every fourth block.
        // With both weight pieces on the lanes a pair of warps shares two blocks: one puts the low pieces' sums into a block,
        // the other adds its own and stores.
        // (64 -> 64 fp32 at 32x32, batch 128: this kernel 39 -> 30 us; without any epilogue it would take 25)
        const int ew = warp - 4, q = ew & 3, part = ew >> 2, pair = part * 2 + (q & 1);
        const float delta = *p.delta_p;
        const int PC = 128 / p.es;
        const bool low = p.split && q >= 2;
        unsigned char *blk = stage + (p.split ? 2 * pair : ew) * kBlock;
        unsigned flip = 0;
        bool ok = true;
        long long it = 0, we = 0;
        for (long long t = t_first; t < p.ntiles; t += t_step, ++it) {
            const int slot = static_cast<int>(it & 1);
            int ci0, b0, y0;
            tile_of(t, ci0, b0, y0);
            ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.acc_full[slot], static_cast<unsigned>(it >> 1) & 1u, p.err_flag, we));
            if (p.split) ok = pair_all(2 + pair, ok);                // the same decision in both warps
            if (!ok) break;
            tc_fence_after();
            const int ci_w = ci0 + (p.split ? (q & 1) : q) * 32;
            const int rows_valid = p.H - y0 < p.Ht ? p.H - y0 : p.Ht, len = rows_valid * p.W, nc = (len + PC - 1) / PC;
            const int nblk = ci_w < p.Cin ? nc * (p.B - b0 < p.nb ? p.B - b0 : p.nb) : 0;
            const unsigned acc = tmem_base + (static_cast<unsigned>(q * 32) << 16) + slot * kAccCols;
            for (int k = part; k < nblk; k += PARTS) {
                const int img = k / nc, i0 = (k - img * nc) * PC;
                unsigned v[32];
                load_positions(acc + img * p.img_rows, i0, len, p, v);
                unsigned char *row = blk + flip * kBlock + lane * 128;
                if (!low) {
                    if (lane == 0) bulk_wait_read_all();             // what was stored before has been read
                    __syncwarp();
                }
                if (p.split) {
                    if (low) {
#pragma unroll
                        for (int h = 0; h < 8; ++h)
                            *reinterpret_cast<uint4 *>(row + ((h ^ (lane & 7)) << 4)) = make_uint4(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
                    }
                    pair_sync(2 + pair);
                    flip ^= 1u;
                    if (low) continue;
#pragma unroll
                    for (int h = 0; h < 8; ++h) {
                        float4 *at = reinterpret_cast<float4 *>(row + ((h ^ (lane & 7)) << 4));
                        const float4 l = *at;
                        *at = make_float4((__uint_as_float(v[4 * h]) + l.x) * delta, (__uint_as_float(v[4 * h + 1]) + l.y) * delta,
                                          (__uint_as_float(v[4 * h + 2]) + l.z) * delta, (__uint_as_float(v[4 * h + 3]) + l.w) * delta);
                    }
                } else if (p.es == 4) {
#pragma unroll
                    for (int h = 0; h < 8; ++h)
                        *reinterpret_cast<float4 *>(row + ((h ^ (lane & 7)) << 4)) =
                            make_float4(__uint_as_float(v[4 * h]) * delta, __uint_as_float(v[4 * h + 1]) * delta,
                                        __uint_as_float(v[4 * h + 2]) * delta, __uint_as_float(v[4 * h + 3]) * delta);
                } else {
#pragma unroll
                    for (int half = 0; half < 2; ++half) {
                        if (half) load_positions(acc + img * p.img_rows, i0 + 32, len, p, v);
#pragma unroll
                        for (int h = 0; h < 4; ++h) {
                            unsigned w[4];
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[8 * h + 2 * e]) * delta,
                                                                                __uint_as_float(v[8 * h + 2 * e + 1]) * delta);
                                w[e] = *reinterpret_cast<const unsigned *>(&b2);
                            }
                            *reinterpret_cast<uint4 *>(row + (((4 * half + h) ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                        }
                    }
                }
                fence_async_proxy();
                __syncwarp();
                if (lane == 0) {                                     // what lies outside the tensor (or the patch) is skipped
                    if (rows_valid == p.Ht) tma_store_4d(&map_o, i0, y0 / p.Ht, ci_w, b0 + img, row);
                    else tma_store_4d(&map_t, y0 * p.W + i0, 0, ci_w, b0 + img, row);
                    bulk_commit();
                }
            }
            tc_fence_before();
            warp_arrive(&pipe.acc_empty[slot]);
        }
        if (lane == 0) bulk_wait_read_all();
        if (ew == 0 && lane == 0) report_wait(p.stats, 5, we);
    } else {
        // epilogue: TMEM lane = input channel, column = patch position. Warp (q, part): lane quarter q,
        // its share of the 32-column chunks.
        const int ew = warp - 4, q = ew & 3, part = ew >> 2;
        const int et = threadIdx.x - 128;                           // 0 .. 511
        const float delta = *p.delta_p;
        const int nchunk = (p.N + 31) >> 5, ch_lo = (nchunk * part + PARTS - 1) >> (LEAN ? 1 : 2), ch_hi = (nchunk * (part + 1) + PARTS - 1) >> (LEAN ? 1 : 2);
        const int HW = p.H * p.W;
        bool ok = true;
        long long it = 0;
        long long we = 0;
        for (long long t = t_first; t < p.ntiles; t += t_step, ++it) {
            const int slot = static_cast<int>(it & 1);
            const unsigned uses = static_cast<unsigned>(it >> 1);
            int ci0, b0, y0;
            tile_of(t, ci0, b0, y0);
            ok = epilogue_all<kEpiThreads>(mbar_wait_timed(&pipe.acc_full[slot], uses & 1u, p.err_flag, we));
            if (!ok) break;                                          // the same decision in every epilogue thread
            tc_fence_after();
            const int ci_l = q * 32 + lane;
            const int rows_valid = p.H - y0 < p.Ht ? p.H - y0 : p.Ht;
            // ---- phase A: accumulator -> staging block (rows of bf16 or fp32 values per channel)
            if (ci0 + (p.split ? (q & 1) * 32 : q * 32) < p.Cin) {   // warp-uniform: some of my 32 channels exist
                unsigned char *row = stage + ci_l * p.pitch;
                for (int chn = ch_lo; chn < ch_hi; ++chn) {
                    unsigned v[32];
                    tmem_ld32(tmem_base + (static_cast<unsigned>(q * 32) << 16) + slot * kAccCols + chn * 32, v);
                    const short *off = s_off + chn * 32;
                    // the 32 table entries of the chunk as four 16-byte loads
                    const uint4 *tp = reinterpret_cast<const uint4 *>(off);
                    const uint4 t0 = tp[0], t1 = tp[1], t2 = tp[2], t3 = tp[3];
                    const unsigned tw[16] = {t0.x, t0.y, t0.z, t0.w, t1.x, t1.y, t1.z, t1.w,
                                             t2.x, t2.y, t2.z, t2.w, t3.x, t3.y, t3.z, t3.w};
                    if (p.es == 4 || KS > 1) {
                        const float f = KS > 1 || p.split ? 1.f : delta;      // parts of a sum are scaled when they have met
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int o = static_cast<int>(static_cast<short>((tw[j >> 1] >> (16 * (j & 1))) & 0xffffu));
                            if (o >= 0) *reinterpret_cast<float *>(row + 4 * o) = __uint_as_float(v[j]) * f;
                        }
                    } else if (p.pairs) {
                        // entry 2i tells where columns 2i, 2i+1 go
#pragma unroll
                        for (int i = 0; i < 16; ++i) {
                            const int o = static_cast<int>(static_cast<short>(tw[i] & 0xffffu));
                            const __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v[2 * i]) * delta, __uint_as_float(v[2 * i + 1]) * delta);
                            if (o >= 0) *reinterpret_cast<unsigned *>(row + 2 * o) = *reinterpret_cast<const unsigned *>(&h);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const int o = static_cast<int>(static_cast<short>((tw[j >> 1] >> (16 * (j & 1))) & 0xffffu));
                            if (o >= 0) *reinterpret_cast<__nv_bfloat16 *>(row + 2 * o) = __float2bfloat16_rn(__uint_as_float(v[j]) * delta);
                        }
                    }
                }
            }
            if (KS > 1) continue;                                  // one tile per cluster: the sums meet below
            // the accumulator is free once every epilogue warp has read its part
            tc_fence_before();
            warp_arrive(&pipe.acc_empty[slot]);
            asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
            // ---- phase B: staging block -> dX, runs of consecutive positions per (image, channel)
            {
                const int ncv = p.Cin - ci0 < 128 ? p.Cin - ci0 : 128;
                const int len = rows_valid * p.W;                    // elements per run
                unsigned char *dst0 = static_cast<unsigned char *>(p.dX);
                const bool words = p.es == 4 || p.pairs;             // whole 32-bit words
                const int nwords = p.es == 4 ? len : len >> 1;
                for (int img = 0; img < p.nb && b0 + img < p.B; ++img) {
                    for (int r = et >> 5; r < ncv; r += kEpiThreads / 32) {
                        const unsigned char *src = stage + r * p.pitch + p.es * img * p.run;
                        unsigned char *dst = dst0 + ((static_cast<long long>(b0 + img) * p.Cin + ci0 + r) * HW + y0 * p.W) * p.es;
                        // four independent loads per lane and round: one by one the round trips through shared memory
                        // were what an epilogue took its time for
                        if (p.split) {                           // the low pieces' sums, 64 rows further, and the high pieces'
                            const float *hi = reinterpret_cast<const float *>(src), *lo = reinterpret_cast<const float *>(src + 64 * p.pitch);
                            copy_run(reinterpret_cast<float *>(dst), len, lane, [&](int i) { return (hi[i] + lo[i]) * delta; });
                        } else if (words) {
                            copy_run(reinterpret_cast<unsigned *>(dst), nwords, lane, [&](int i) { return reinterpret_cast<const unsigned *>(src)[i]; });
                        } else {
                            copy_run(reinterpret_cast<unsigned short *>(dst), len, lane,
                                     [&](int i) { return reinterpret_cast<const unsigned short *>(src)[i]; });
                        }
                    }
                }
            }
            // the staging block is rewritten by the next tile only after everyone is done reading it
            asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory");
        }
        if (et == 0) report_wait(p.stats, 5, we);
    }
    if (KS > 1) {
        cluster_barrier();                 // every CTA's partial sums are staged
        // this CTA finishes 128 / KS channels: rows read from all staging blocks, lanes along the positions
        int ci0, b0, y0;
        tile_of(t_first, ci0, b0, y0);
        const int per = 128 / KS, rows_valid = p.H - y0 < p.Ht ? p.H - y0 : p.Ht, len = rows_valid * p.W, HW = p.H * p.W;
        const int nimg = p.B - b0 < p.nb ? p.B - b0 : p.nb, row_len = (nimg - 1) * p.run + len;
        const float delta = *p.delta_p;
        unsigned base[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < KS) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base[k]) : "r"(smem_u32(stage)), "r"(k));
        for (int r = warp; r < per; r += kThreadsX / 32) {
            const int cl = rank * per + r, ci = ci0 + cl;
            if (ci >= p.Cin) break;
            for (int i0 = lane; i0 < row_len; i0 += 128) {           // whole images are back to back in the staged row
                float v[4][8];
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k < KS && i0 + 32 * u < row_len)
                            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[u][k]) : "r"(base[k] + cl * p.pitch + 4 * (i0 + 32 * u)));
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = i0 + 32 * u;
                    if (i >= row_len) break;
                    float sum = 0.f;
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k < KS) sum += v[u][k];
                    const int img = i / p.run, pos = i - img * p.run;
                    const long long o = (static_cast<long long>(b0 + img) * p.Cin + ci) * HW + y0 * p.W + pos;
                    if (p.es == 4) static_cast<float *>(p.dX)[o] = sum * delta;
                    else static_cast<__nv_bfloat16 *>(p.dX)[o] = __float2bfloat16_rn(sum * delta);
                }
            }
        }
        cluster_barrier();                 // nobody leaves while its staging block is still being read
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 2) {
        __syncwarp();
        tmem_dealloc(tmem_base, kTmem);
    }
}

// weights [Cout][Cin][3][3] -> [9][Cout][pitch] bf16 (the tap's [co][ci] matrix with ci contiguous, the row pitch a
// multiple of 8). fp32 weights -> [18][Cout][pitch]: taps 0-8 hold the values rounded to bf16, taps 9-17 what that
// rounding left over, rounded to bf16 again. The sum of the two pieces differs from the fp32 value by at most 2^-17 of
// it (2.4e-6 rms), and a code times a piece is exact in the fp32 accumulator. Used when the step size is given; otherwise the
// statistics kernel does this on the side.
template <typename T>
__global__ void __launch_bounds__(256)
w_taps_rows_kernel(const T *__restrict__ W, __nv_bfloat16 *__restrict__ out, long long Cout, long long Cin, long long pitch) {
    chain_wait();
    chain_release();
    constexpr int TAPS = sizeof(T) == 4 ? 18 : 9;
    const long long n = Cout * Cin * 9;
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < n; i += gridDim.x * 256ll) {
        const long long ci = i % Cin, t = (i / Cin) % 9, co = i / (Cin * 9);
        const float w = static_cast<float>(W[(co * Cin + ci) * 9 + t]);
        const __nv_bfloat16 hi = __float2bfloat16_rn(w);
        out[(t * Cout + co) * pitch + ci] = hi;
        if (TAPS == 18) out[((9 + t) * Cout + co) * pitch + ci] = __float2bfloat16_rn(w - __bfloat162float(hi));
    }
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

}  // namespace

// Shapes the TMA-fed 3x3 kernels take. fp32 operands are split into two bf16 pieces each (the codes are exact in bf16);
// rows of the codes, of the re-laid weights and of the activations that are no multiple of 16 bytes are padded to one.
// An fp32 dX keeps to kMaxMmas per accumulator, and its reduction is cut into eight parts at most: longer ones go to the gather
// kernels unless the caller insists on these (a part then has more MMAs than that).
constexpr int kMaxKS = 8;
constexpr int kMaxBlocks = kMaxMmas / 36;        // 64-channel blocks of co per accumulator: nine taps of four MMAs each
bool tc3_tma_supported(const ConvShape &s, int io, bool dx_f32) {
    return (io == DBP_BF16 || io == DBP_F32) && s.k == 3 && s.W >= 1 && s.W <= 62 && s.H <= 4096 && s.B * s.H * s.W < (1ll << 30) &&
           (!dx_f32 || s.Cout <= 64ll * kMaxBlocks * kMaxKS);
}

namespace {
// How a layer's dX is made: patches (t, with no pointers in it) or rows of several images
struct Dx3Plan {
    Dx3T t{};
    size_t smem = 0;
    bool small = false, by_rows = false;
    RowsPlan rows;
    int map_taps = 9;
};

// share: the caller can use the other half of every SM. false: the shape does not fit
bool plan_tc3_dx(const dbp_ctx *ctx, const ConvShape &s, int io, int es, bool share, Dx3Plan &plan) {
    Dx3T p{};
    p.es = es;
    p.ntaps = io == DBP_F32 ? 18 : 9;
    p.B = static_cast<int>(s.B); p.Cin = static_cast<int>(s.Cin); p.Cout = static_cast<int>(s.Cout);
    p.H = static_cast<int>(s.H); p.W = static_cast<int>(s.W);
    p.phase_cin = (ctx->phase_cin > 0 && ctx->phase_cin % 128 == 0 && s.Cin == 4ll * ctx->phase_cin) ? ctx->phase_cin : 0;
    p.ncb = (p.Cout + 63) / 64;
    p.ci_tiles = (p.Cin + 127) / 128;
    // Parts of a long reduction (an fp32 result's: bf16 rounds far coarser than the accumulators do). The two pieces of fp32
    // weights then take a pass each, low ones first, because an MMA costs an accumulator as much for a small term as for a
    // large one: up to kMaxBlocks / 2 blocks the sum of both pieces keeps to kMaxMmas anyway, and a block's codes are read once.
    int min_ks = 1;
    while (p.es == 4 && min_ks < kMaxKS && min_ks * kMaxBlocks < p.ncb) min_ks *= 2;
    p.split = io == DBP_F32 && p.Cin <= 64 && min_ks == 1 ? 1 : 0;
    p.a_panels = p.Cin <= 64 && !p.split ? 1 : 2;
    plan.map_taps = p.ntaps;
    if (p.split) p.ntaps = 9;
    p.nq = kMaxQ;
    const int sms = ctx->sm_count;
    size_t smem = 0;
    double best = 1e300;
    Dx3T chosen{};
    bool small = false;
    int wide_ks = 1;
    // The cheapest of the candidate patches (rows of one image, or several whole images) and reduction splits by a count of
    // clocks (see the head of this file; 6 KB per clock is about what the L2 delivers to all SMs together). Returns whether the
    // patch still fits the accumulator.
    auto consider = [&](int ht, int nb, int ks) -> bool {
        Dx3T q = p;
        q.Ht = ht; q.nb = nb; q.KS = ks;
        const int cbs = (p.ncb + ks - 1) / ks;
        q.passes = p.ntaps == 18 && 2 * cbs > kMaxBlocks ? 2 : 1;
        q.tiles_y = (p.H + ht - 1) / ht;
        q.run = ht * p.W;
        // by the copy engine where every run starts on 16 bytes, a row is whole words of at least four columns (tensor memory
        // is read in pieces of a row) and a run fills a block
        const int hw = p.H * p.W, low_bit = p.W & -p.W;
        q.unit = ks == 1 && low_bit >= 4 && hw * p.es % 16 == 0 && (q.tiles_y == 1 || q.run * p.es % 16 == 0) && q.run * p.es >= 128
                     ? (low_bit > 32 ? 32 : low_bit) : 0;
        q.w_rcp = (65536u + p.W - 1) / p.W;
        q.Wp = (p.W % 2 == 0 && p.es == 2 && ks == 1 && q.unit == 0) ? p.W + 2 : p.W + 1;
        q.img_rows = (nb == 1 ? ht + 2 : ht + 1) * q.Wp;
        q.N = round_up((nb - 1) * q.img_rows + (ht - 1) * q.Wp + p.W, 16);    // up to the last column that holds an output
        if (q.N > 256) return false;
        const int rows_read = q.N + 2 * q.Wp + 2;
        q.q_bytes = round_up((rows_read > q.img_rows * nb ? rows_read : q.img_rows * nb) * 128, 1024);
        q.q_tx = q.img_rows * nb * 128;
        q.pos_tiles = nb == 1 ? static_cast<long long>(p.B) * q.tiles_y : (p.B + nb - 1) / nb;
        q.ntiles = q.pos_tiles * p.ci_tiles;
        // one round of clusters; a GPC's SMs are no multiple of 4 or 8, so not all of them can be covered (36 clusters of 4
        // took 39 us where 32 took 24)
        if (ks > min_ks && q.ntiles * ks > (ks == 2 ? sms : ks == 4 ? sms * 7 / 8 : sms * 3 / 4)) return true;
        if (small && (q.ntiles * ks > sms || ks != wide_ks)) return true;      // (the order of a sum does not depend on what else is asked for)
        // an odd number of 32-bit words per row: the 32 channels of a warp hit 32 different banks when they stage the same
        // position
        const int es = ks > 1 ? 4 : p.es;
        q.pitch = round_up(nb * q.run * es, 4);
        if ((q.pitch / 4) % 2 == 0) q.pitch += 4;
        q.pairs = p.W % 2 == 0 ? 1 : 0;
        // Weights: a slot holds G taps and is handed over with one barrier (the hand-over, not the copy instruction, is what
        // costs time). With one ci block and room for all taps of all co blocks they are loaded once and stay; otherwise they
        // stream through a ring of slots.
        const size_t tap_bytes = static_cast<size_t>(p.a_panels) * kWPanel, budget = small ? kHalfSm : 227 * 1024 - 2048;
        const size_t rings = static_cast<size_t>(q.nq) * q.q_bytes;
        const size_t staging = (q.unit > 0 ? static_cast<size_t>(small ? kEpiWarps<true> : kEpiWarps<false>) * kBlock : static_cast<size_t>(128) * q.pitch);
        const size_t fixed = rings + (small ? 0 : staging) + 512 + 1024;
        if (small && staging + 512 + 1024 > budget) return true;
        if (fixed + 3 * tap_bytes > budget) return true;
        const size_t room = budget - fixed;
        const int slots_all = p.ncb * (p.ntaps / 9);
        if (p.phase_cin > 0) {
            q.resident = 0; q.G = 2; q.nw = static_cast<int>(room / (2 * tap_bytes));
            if (q.nw < 2) return true;
        } else if (ks == 1 && p.ci_tiles == 1 && slots_all <= kMaxW && static_cast<size_t>(slots_all) * 9 * tap_bytes <= room) {
            q.resident = 1; q.G = 9; q.nw = slots_all;
        } else if (room >= 2 * 3 * tap_bytes) {
            q.resident = 0; q.G = 3; q.nw = static_cast<int>(room / (3 * tap_bytes));
        } else {
            q.resident = 0; q.G = 1; q.nw = static_cast<int>(room / tap_bytes);
        }
        if (q.nw > kMaxW) q.nw = kMaxW;
        q.w_slot = static_cast<int>(q.G * tap_bytes);
        q.slots = (p.phase_cin > 0 ? p.ntaps / 9 : p.ntaps / q.G) / q.passes;
        const double live = p.phase_cin > 0 ? 0.25 : 1.0;
        const long long ctas = q.ntiles * ks, waves = (ctas + sms - 1) / sms, active = ctas < sms ? ctas : sms;
        double mma = 32.0 + 0.25 * q.N + (q.resident ? 0.0 : 16.0 * p.a_panels);
        if (mma < 0.5 * q.N) mma = 0.5 * q.N;
        const double l2 = q.resident ? 0.0 : 2048.0 * p.a_panels * static_cast<double>(active) / 6000.0;
        if (mma < l2) mma = l2;
        const double body = cbs * (p.ntaps * live * 4.0 * mma + (q.resident ? 0.0 : 250.0 * (p.phase_cin > 0 ? p.ntaps / 6.0 : static_cast<double>(p.ntaps) / q.G)) + q.passes * (q.q_tx / 128.0 + 300.0));
        const double staged = (p.Cin <= 64 && !p.split ? 64.0 : 128.0) * nb * q.run * es;
        const double epi = (q.unit > 0 ? 1000.0 + staged / 40.0 : 2000.0 + staged / 20.0) + (ks > 1 ? 2000.0 + staged / 8.0 : 0.0);
        const double cost = static_cast<double>(waves) * (500.0 + (body > epi ? body : epi)) + (waves > 1 ? (body < epi ? body : epi) : epi);
        if (cost < best) {
            best = cost;
            const size_t operands = rings + static_cast<size_t>(q.nw) * q.w_slot, over = operands > staging ? operands : staging;
            q.off_at = static_cast<int>(small ? over : operands + staging);
            chosen = q;
            smem = q.off_at + 512 + 1024;
        }
        return true;
    };
    auto search = [&] {
        for (int ht = 1; ht <= p.H; ++ht)
            if (!consider(ht, 1, min_ks)) break;
        for (int ks = min_ks; ks <= kMaxKS; ks *= 2) {
            if (ks > p.ncb || (ks > 1 && p.split)) break;
            for (int nb = ks > 1 ? 1 : 2; nb <= 64 && nb <= p.B; ++nb)
                if (!consider(p.H, nb, ks)) break;
        }
    };
    search();
    if (smem == 0) return false;
    // Rows of several images instead of patches (tc3_rows_dx.cu), by the same count of clocks and whatever else is asked for, because
    // the order of a sum depends on the way it is made: tiles that fit half an SM where they take less than 0.85, wider ones,
    // beside which no dW CTA fits, where they take less than 0.65. dX alone and the joined call, us, patches against rows, by the ratio of the counts:
    // 0.60 512 -> 512 fp32 at 2x2, batch 128: 29.2, 21.0; 52.1, 48.7; 0.59 at 4x4: 45.3, 30.6; 75.1, 68.1; 0.70 256 -> 512 at 4x4: 31.6, 23.6;
    // 49.0, 44.2; 0.73 128 -> 256 at 8x8: 33.2, 26.6; 47.7, 40.3 (wide: 25.5, 51.2); 0.85 bf16 768 -> 384 at 3x4, batch 70: 29.5, 25.7;
    // 65.8, 57.8; 0.86 512 -> 512 at 7x7, batch 64: 36.6, 41.4; 67.9, 69.3; 0.91 256 -> 256 fp32 at 8x8, batch 128: 34.4, 34.8; 54.3, 53.9.
    RowsPlan rows_wide, &rows_plan = plan.rows;
    const int weight_pieces = io == DBP_F32 ? 2 : 1;
    const double rows_cost = tc3_rows_plan(ctx, s, weight_pieces, kRowsLeanCols, &rows_plan);
    bool &by_rows = plan.by_rows;
    if (rows_cost > 0) {
        double patches = best;
        if (p.es == 2) {                         // decided for an fp32 dX, so that the bf16 one is that one rounded
            const Dx3T found = chosen;
            const size_t found_smem = smem;
            p.es = 4;
            best = 1e300;
            search();
            p.es = 2;
            patches = best;
            chosen = found;
            smem = found_smem;
        }
        by_rows = rows_cost < 0.85 * patches;
        const double wide_cost = tc3_rows_plan(ctx, s, weight_pieces, kRowsMaxCols, &rows_wide);
        if (wide_cost < 0.65 * patches && wide_cost < rows_cost) {
            by_rows = true;
            rows_plan = rows_wide;
        }
    }
    // Half an SM's worth of it, when the caller can use the other half: only with one round of CTAs (then the staging block can
    // lie over the operands), and not for phase images, whose slots of two taps do not fit
    const bool one_wave = chosen.ntiles * chosen.KS <= sms;
    if (share && one_wave && p.phase_cin == 0 && !by_rows) {
        const Dx3T wide = chosen;
        const size_t wide_smem = smem;
        small = true;
        wide_ks = wide.KS;
        best = 1e300;
        smem = 0;
        search();
        small = smem != 0;
        if (!small) { chosen = wide; smem = wide_smem; }
    }
    plan.small = small;
    plan.t = chosen;
    plan.smem = smem;
    return true;
}

// The search is a microsecond of divisions on the host, of the twenty that a small layer's call is bound by (bf16 128 -> 128 at 7x7,
// batch 8, joined: 20.2 us of host time without the kept plans, 19.1 with). A thread keeps the plans of the shapes it saw last.
const Dx3Plan *plan_of(const dbp_ctx *ctx, const ConvShape &s, int io, int es, bool share) {
    struct Entry {
        ConvShape s{};
        int io = 0, es = 0, phase_cin = 0, sms = 0;
        bool share = false, fits = false;
        Dx3Plan plan;
    };
    constexpr int kKept = 32;
    static thread_local Entry kept[kKept];
    static thread_local int count = 0, next = 0;
    for (int i = 0; i < count; ++i) {
        const Entry &e = kept[i];
        if (e.s.B == s.B && e.s.Cin == s.Cin && e.s.Cout == s.Cout && e.s.H == s.H && e.s.W == s.W && e.io == io && e.es == es &&
            e.share == share && e.phase_cin == ctx->phase_cin && e.sms == ctx->sm_count)
            return e.fits ? &e.plan : nullptr;
    }
    Entry &e = kept[next];
    next = (next + 1) % kKept;
    if (count < kKept) ++count;
    e = Entry{};
    e.s = s; e.io = io; e.es = es; e.share = share; e.phase_cin = ctx->phase_cin; e.sms = ctx->sm_count;
    e.fits = plan_tc3_dx(ctx, s, io, es, share, e.plan);
    return e.fits ? &e.plan : nullptr;
}
}  // namespace

// DBP_EUNSUPPORTED: the shape does not fit (the caller uses another kernel)
int launch_tc3_tma_dx(dbp_ctx *ctx, const void *codes_nhwc, const void *W, int io, const float *delta_p,
                      const ConvShape &s, void *dX, bool dx_bf16, int *err_flag, bool weights_ready, bool *lean) {
    if (!tc3_tma_supported(s, io, false)) return DBP_EUNSUPPORTED;
    const Dx3Plan *const plan = plan_of(ctx, s, io, dx_bf16 ? 2 : 4, lean != nullptr);
    if (plan == nullptr) return DBP_EUNSUPPORTED;
    Dx3T p = plan->t;
    p.delta_p = delta_p; p.dX = dX; p.err_flag = err_flag; p.stats = ctx->wait_stats;
    const bool small = plan->small;
    const size_t smem = plan->smem;
    const int map_taps = plan->map_taps, sms = ctx->sm_count;
    if (lean != nullptr) *lean = small;

    // re-laid weights
    const long long w_pitch = (s.Cin + 7) / 8 * 8, q_pitch = (s.Cout + 7) / 8 * 8;
    const size_t wb = sizeof(__nv_bfloat16) * static_cast<size_t>(s.Cout) * w_pitch * map_taps;
    int rc = ws_reserve(ctx, ctx->w_taps, wb);
    if (rc) return rc;
    if (!weights_ready) {
        long long blocks = (static_cast<long long>(s.Cout) * s.Cin * 9 + 255) / 256;
        if (blocks > sms * 8) blocks = sms * 8;
        __nv_bfloat16 *taps = static_cast<__nv_bfloat16 *>(ctx->w_taps.ptr);
        if (io == DBP_F32)
            rc = cuda_ok(launch_chained(w_taps_rows_kernel<float>, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, ctx->stream,
                                        static_cast<const float *>(W), taps, s.Cout, s.Cin, w_pitch));
        else
            rc = cuda_ok(launch_chained(w_taps_rows_kernel<__nv_bfloat16>, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, ctx->stream,
                                        static_cast<const __nv_bfloat16 *>(W), taps, s.Cout, s.Cin, w_pitch));
        if (rc) return rc;
    }
    if (plan->by_rows) return launch_tc3_rows_dx(ctx, plan->rows, codes_nhwc, io == DBP_F32 ? 2 : 1, delta_p, s, dX, dx_bf16, err_flag, lean);
    CUtensorMap map_q, map_w;
    {
        const unsigned long long dims[4] = {static_cast<unsigned long long>(s.Cout), static_cast<unsigned long long>(s.W),
                                            static_cast<unsigned long long>(s.H), static_cast<unsigned long long>(s.B)};
        const unsigned long long row = static_cast<unsigned long long>(q_pitch) * 2;
        const unsigned long long str[3] = {row, row * s.W, row * s.W * s.H};
        const unsigned box[4] = {64, static_cast<unsigned>(p.Wp), static_cast<unsigned>(p.img_rows / p.Wp), static_cast<unsigned>(p.nb)};
        if (!encode_map_bf16(&map_q, codes_nhwc, 4, dims, str, box)) return fail_cuda("tensor map of the code patches");
    }
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(s.Cin), static_cast<unsigned long long>(s.Cout),
                                            static_cast<unsigned long long>(map_taps)};
        const unsigned long long str[2] = {static_cast<unsigned long long>(w_pitch) * 2,
                                           static_cast<unsigned long long>(w_pitch) * 2 * s.Cout};
        const unsigned box[3] = {64, 64, static_cast<unsigned>(p.phase_cin > 0 ? 1 : p.G)};
        if (!encode_map_bf16(&map_w, ctx->w_taps.ptr, 3, dims, str, box)) return fail_cuda("tensor map of the weights");
    }
    CUtensorMap map_o = map_q, map_t = map_q;
    if (p.unit > 0) {
        // dX as [b][ci][patch][positions of a patch], and as [b][ci][positions] for a last patch of fewer rows
        const unsigned long long HW = static_cast<unsigned long long>(s.H) * s.W, plane = HW * p.es, full = static_cast<unsigned long long>(s.H / p.Ht);
        const unsigned long long dims_o[4] = {static_cast<unsigned long long>(p.run), full, static_cast<unsigned long long>(s.Cin), static_cast<unsigned long long>(s.B)};
        const unsigned long long dims_t[4] = {HW, 1, static_cast<unsigned long long>(s.Cin), static_cast<unsigned long long>(s.B)};
        const unsigned long long str_o[3] = {full > 1 ? static_cast<unsigned long long>(p.run) * p.es : plane, plane, plane * s.Cin};
        const unsigned long long str_t[3] = {plane, plane, plane * s.Cin};
        const unsigned box[4] = {static_cast<unsigned>(128 / p.es), 1, 32, 1};
        auto encode = p.es == 4 ? encode_map_f32_sw128 : encode_map_bf16;
        if (!encode(&map_o, dX, 4, dims_o, str_o, box) || !encode(&map_t, dX, 4, dims_t, str_t, box)) return fail_cuda("tensor map of dX");
    }
    auto kern = small ? (p.unit > 0 ? tc3_tma_dx_kernel<true, true> : tc3_tma_dx_kernel<false, true>)
                      : (p.unit > 0 ? tc3_tma_dx_kernel<true, false> : tc3_tma_dx_kernel<false, false>);
    const int threads = small ? kThreads3<true> : kThreads3<false>;
    if (small) cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (allow_shared(kern) != cudaSuccess)
        return fail_cuda("shared memory size");
    if (p.KS > 1)
        return cuda_ok(launch_chained_cluster(kern, static_cast<unsigned>(p.ntiles) * p.KS, static_cast<unsigned>(p.KS),
                                              dim3(threads), smem, ctx->stream, map_q, map_w, map_o, map_t, p));
    const long long grid = p.ntiles < sms ? p.ntiles : sms;
    return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(grid)), dim3(threads), smem, ctx->stream,
                                  map_q, map_w, map_o, map_t, p));
}

}  // namespace dbp
