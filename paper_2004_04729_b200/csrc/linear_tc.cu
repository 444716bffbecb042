// Both products of a linear layer on the tensor cores in one launch (Eqs. (qda), (qdw)):
//   dX[b, k] = Delta * sum_j q[b, j] W[j, k]        dW[j, k] = Delta * sum_b q[b, j] X[b, k]
// The codes lie row-major as bf16 [B][pitch], X and W row-major [rows][K] in bf16 (fp32 operands as two bf16
// pieces, one tensor after the other: the reduction then runs over both pieces with the codes read twice). Both
// products are [M x cols] = A * B with the reduction index as the row of B:
//   dX: A = codes [128 b][64 j]   K-major          B = W [64 j][k ...]   MN-major
//   dW: A = codes [64 b][128 j]   MN-major         B = X [64 b][k ...]   MN-major
// so every operand tile is one or a few tiled copies of row-major memory, and one kernel runs the tiles of both
// products: their CTAs fill the GPU together, and neither product waits for the other's last wave.
//
// A CTA is persistent over output tiles of 128 MA rows x TN columns: warp 0 issues the copies, warp 1 the MMAs into
// one of two accumulators in tensor memory (MA = 2: both are one tile's), warps 2-9 drain the other one (scale by Delta,
// convert, stage as 128-byte swizzled rows, one tiled store per 32-row block; rows whose pitch is no multiple of 16 bytes
// leave through plain stores). Weight-gradient tiles may be split along the reduction: the parts then add into a
// cleared dW through the copy engine.
// Large layers are bound by what the copies bring to an SM, about 60 bytes a clock: a step of 128 x 256 x 64 is 512 clocks of
// the tensor pipe and 48 KB (840 clocks measured), one of 256 x 256 x 64 1024 clocks and 64 KB. Small ones are bound by the
// chain of reduction steps of the CTA with the most of them (linear_plan), and a step by its hand-overs, so the issuing loops
// carry no divisions. 1024 -> 4096 bf16, batch 4096: the call 95.0 -> 84.7 us; 2048 -> 1000 fp32, batch 256: 32.1 -> 23.7.
#include "tc_common.cuh"

#include <utility>

namespace dbp {

namespace {

using namespace tc;

constexpr int kStagesL = 8;                      // most stages of the ring (narrow tiles)
constexpr int kPanelL = 64 * 128;                // 64 rows x 128 bytes
constexpr int kABytesL = 2 * kPanelL;            // 128 x 64 bf16 either way round
constexpr int kMaxNL = 256;
constexpr int kRingL = 4 * (kABytesL + (kMaxNL / 64) * kPanelL);     // bytes of the ring: four stages of the widest tile
constexpr int kEpiWarpsL = 8;
constexpr int kThreadsL = 64 + 32 * kEpiWarpsL;
constexpr int kOutBlock = 32 * 128;              // one warp's staged block: 32 rows of 128 bytes

struct LinProduct {
    void *out;                    // [M][cols], fp32 or bf16
    int out_f32, tma_out, add;    // add: into an fp32 output that was cleared, or that holds the part of the reduction before this one
    int M, cols;
    int a_kmajor;                 // A is [M][reduction] (dX) instead of [reduction][M] (dW)
    int ks, pieces, steps;        // 64-deep steps per piece; steps of all pieces
    int per_split, nsplit;
    int mt;                       // tiles of 128 MA rows
    int tiles;                    // mt * column tiles * nsplit
};

struct LinArgs {
    LinProduct pr[2];             // the product with the longer tiles first
    int nprod, tiles, TN, MA;     // MA accumulators of 128 rows per tile: with two, both are one tile's
    int lead;                     // tiles of the second product for a CTA that has one tile less of the first: see tile_at
    int stages, stage_bytes;      // as many stages as the ring holds: a narrow tile's steps are bound by the copies' latency
    const float *delta_p;
    int *err_flag;
};

struct LinMaps {
    CUtensorMap a[2], b[2], out[2];
};

struct PipeL {
    unsigned long long full[kStagesL], empty[kStagesL], acc_full[2], acc_empty[2];
    unsigned tmem_base;
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int c0, int c1, const void *src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(map), "r"(c0), "r"(c1), "r"(smem_u32(src)) : "memory");
}

template <int MA>
__global__ void __launch_bounds__(kThreadsL, 1)
linear_products_kernel(const __grid_constant__ LinMaps maps, const __grid_constant__ LinArgs p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ PipeL pipe;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = p.stages, stage_bytes = p.stage_bytes;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&pipe.full[s], 1);
            mbar_init(&pipe.empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&pipe.acc_full[a], 1);
            mbar_init(&pipe.acc_empty[a], kEpiWarpsL);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int i = 0; i < p.nprod; ++i) {
            tma_prefetch_desc(&maps.a[i]);
            tma_prefetch_desc(&maps.b[i]);
            if (p.pr[i].tma_out) tma_prefetch_desc(&maps.out[i]);
        }
    }
    if (warp == 1) tmem_alloc(&pipe.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = pipe.tmem_base;
    chain_wait();        // from here on the kernel reads what earlier kernels wrote
    chain_release();

    // This CTA's tile number j: product, first row and column, range of reduction steps. The longer tiles (the first product's)
    // are dealt in turn; a CTA that got one less of them takes `lead` of the shorter ones, which last as long, before these go
    // around, from the last CTA down.
    const int G = static_cast<int>(gridDim.x), cta = static_cast<int>(blockIdx.x);
    const int n0_tiles = p.pr[0].tiles, n1_tiles = p.tiles - n0_tiles, more = n0_tiles % G, mine = (n0_tiles - cta + G - 1) / G;
    struct Tile { int i, m0, n0, k0, k1, na; };
    auto tile_at = [&](int j, Tile &r) {
        int t = cta + j * G;
        if (t >= n0_tiles) {
            j -= mine;
            if (cta >= more && j < p.lead) t = cta - more + j * (G - more);
            else t = p.lead * (G - more) + G - 1 - cta + (j - (cta >= more ? p.lead : 0)) * G;
            if (t >= n1_tiles) return false;
            t += n0_tiles;
        }
        r.i = t < p.pr[0].tiles ? 0 : 1;
        const LinProduct &q = p.pr[r.i];
        if (r.i) t -= p.pr[0].tiles;
        const int s = t % q.nsplit;
        t /= q.nsplit;
        r.m0 = (t % q.mt) * 128 * MA;
        r.n0 = (t / q.mt) * p.TN;
        r.k0 = s * q.per_split;
        r.k1 = r.k0 + q.per_split < q.steps ? r.k0 + q.per_split : q.steps;
        r.na = MA == 2 && q.M - r.m0 > 128 ? 2 : 1;                  // accumulators that hold rows
        return true;
    };
    Tile tl;

    if (warp == 0) {
        int s = 0;
        unsigned parity = 1;                     // a fresh barrier passes a wait on the previous phase
        bool ok = true;
        for (int it = 0; ok && tile_at(it, tl); ++it) {
            const LinProduct &q = p.pr[tl.i];
            const int left = (q.cols - tl.n0 + 63) >> 6;
            const int nb = left < p.TN / 64 ? left : p.TN / 64;      // 64-column panels that hold columns
            const unsigned tx = static_cast<unsigned>(tl.na * kABytesL + nb * kPanelL);
            const CUtensorMap *const map_a = &maps.a[tl.i], *const map_b = &maps.b[tl.i];
            // the low pieces first: the accumulator is still small when they are added
            int piece = q.pieces - 1 - tl.k0 / q.ks, r0 = tl.k0 % q.ks * 64;
            for (int k = tl.k0; k < tl.k1; ++k) {
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.empty[s], parity, p.err_flag));
                if (!ok) break;
                if (elect_one()) {
                    unsigned char *st = smem + s * stage_bytes;
                    mbar_expect_tx(&pipe.full[s], tx);
#pragma unroll
                    for (int a = 0; a < MA; ++a) {
                        if (a >= tl.na) break;
                        const int m = tl.m0 + 128 * a;
                        if (q.a_kmajor) {
                            tma_load_2d(st + a * kABytesL, map_a, r0, m, &pipe.full[s]);
                        } else {
                            tma_load_2d(st + a * kABytesL, map_a, m, r0, &pipe.full[s]);
                            tma_load_2d(st + a * kABytesL + kPanelL, map_a, m + 64, r0, &pipe.full[s]);
                        }
                    }
                    st += MA * kABytesL;
#pragma unroll
                    for (int i = 0; i < kMaxNL / 64; ++i)
                        if (i < nb) tma_load_3d(st + i * kPanelL, map_b, tl.n0 + 64 * i, r0, piece, &pipe.full[s]);
                }
                if ((r0 += 64) == 64 * q.ks) { r0 = 0; --piece; }
                if (++s == S) { s = 0; parity ^= 1u; }
            }
        }
    } else if (warp == 1) {
        const unsigned idesc_k = make_idesc(128, p.TN, false, true), idesc_mn = make_idesc(128, p.TN, true, true);
        int s = 0;
        unsigned parity = 0;
        bool ok = true;
        for (int it = 0; ok && tile_at(it, tl); ++it) {
            const bool kmaj = p.pr[tl.i].a_kmajor != 0;
            // this tile's accumulator (the first of two) and how often it has been used before
            const int slot = MA == 2 ? 0 : it & 1;
            const unsigned uses = static_cast<unsigned>(MA == 2 ? it : it >> 1);
            const unsigned tmem_d = tmem_base + slot * kMaxNL;
            for (int k = tl.k0; k < tl.k1 && ok; ++k) {
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.full[s], parity, p.err_flag));
                if (!ok) break;
                const unsigned a_addr = smem_u32(smem + s * stage_bytes);
                const unsigned long long bd = make_desc(a_addr + MA * kABytesL, kPanelL, 1024);
#pragma unroll
                for (int a = 0; a < MA; ++a) {
                    if (k == tl.k0) ok = ok && __all_sync(0xffffffffu, mbar_wait(&pipe.acc_empty[slot + a], (uses & 1u) ^ 1u, p.err_flag));
                    if (!ok) break;
                    tc_fence_after();
                    if (elect_one()) {
                        if (a < tl.na) {
                            const unsigned long long ad = make_desc(a_addr + a * kABytesL, kmaj ? 16 : kPanelL, 1024);
                            if (kmaj) {
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk)       // 16 along the rows of A = 32 bytes
                                    mma_bf16(tmem_d + a * kMaxNL, ad + 2 * kk, bd + 128 * kk, idesc_k, (k > tl.k0 || kk > 0) ? 1u : 0u);
                            } else {
#pragma unroll
                                for (int kk = 0; kk < 4; ++kk)       // 16 rows of A = 2048 bytes
                                    mma_bf16(tmem_d + a * kMaxNL, ad + 128 * kk, bd + 128 * kk, idesc_mn, (k > tl.k0 || kk > 0) ? 1u : 0u);
                            }
                        }
                        if (a == MA - 1) mma_commit(&pipe.empty[s]);
                        if (k == tl.k1 - 1) mma_commit(&pipe.acc_full[slot + a]);
                    }
                }
                if (++s == S) { s = 0; parity ^= 1u; }
            }
        }
    } else {
        // epilogue: TMEM lane = output row, column = output column; two warps per lane quarter take turns at the
        // blocks of 32 fp32 or 64 bf16 columns (128 bytes of a row)
        const int q4 = warp & 3, part = (warp - 2) >> 2;
        unsigned char *stage = smem + kRingL + (warp - 2) * kOutBlock;
        const float delta = *p.delta_p;
        bool ok = true;
        for (int it = 0; ok && tile_at(it, tl); ++it) {
          const LinProduct &q = p.pr[tl.i];
          for (int am = 0; am < MA; ++am) {
            const int slot = MA == 2 ? am : it & 1;
            ok = mbar_wait(&pipe.acc_full[slot], static_cast<unsigned>(MA == 2 ? it : it >> 1) & 1u, p.err_flag);
            if (!ok) break;
            tc_fence_after();
            const int row_w = tl.m0 + am * 128 + q4 * 32;          // first output row of this warp
            const int ncol = q.cols - tl.n0 < p.TN ? q.cols - tl.n0 : p.TN;
            const int bw = q.out_f32 ? 32 : 64;                    // columns per block
            if (row_w < q.M) {
                for (int c = part * bw; c < ncol; c += 2 * bw) {
                    const unsigned taddr = tmem_base + (static_cast<unsigned>(q4 * 32) << 16) + slot * kMaxNL + c;
                    unsigned v[32];
                    tmem_ld32(taddr, v);
                    if (lane == 0) bulk_wait_read_all();           // the block's previous store has been read
                    __syncwarp();
                    if (q.out_f32) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            *reinterpret_cast<float4 *>(stage + lane * 128 + ((j ^ (lane & 7)) << 4)) =
                                make_float4(__uint_as_float(v[4 * j]) * delta, __uint_as_float(v[4 * j + 1]) * delta,
                                            __uint_as_float(v[4 * j + 2]) * delta, __uint_as_float(v[4 * j + 3]) * delta);
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h) tmem_ld32(taddr + 32, v);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                unsigned w[4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(v[8 * j + 2 * i]) * delta,
                                                                                    __uint_as_float(v[8 * j + 2 * i + 1]) * delta);
                                    w[i] = *reinterpret_cast<const unsigned *>(&b2);
                                }
                                *reinterpret_cast<uint4 *>(stage + lane * 128 + (((4 * h + j) ^ (lane & 7)) << 4)) =
                                    make_uint4(w[0], w[1], w[2], w[3]);
                            }
                        }
                    }
                    if (q.tma_out) {                               // rows and columns outside the tensor are skipped
                        fence_async_proxy();
                        __syncwarp();
                        if (lane == 0) {
                            if (q.add) tma_reduce_add_2d(&maps.out[tl.i], tl.n0 + c, row_w, stage);
                            else tma_store_2d(&maps.out[tl.i], tl.n0 + c, row_w, stage);
                            bulk_commit();
                        }
                    } else {
                        __syncwarp();
                        // lanes along the columns, eight rows at a time; bf16 as words, shifted by one column in the rows that
                        // start between words
                        const int nr = q.M - row_w < 32 ? q.M - row_w : 32;
                        const int nc = ncol - c < bw ? ncol - c : bw;
                        const long long o0 = static_cast<long long>(row_w) * q.cols + tl.n0 + c;
                        for (int r0 = 0; r0 < nr; r0 += 8) {
                            unsigned x[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                x[i] = *reinterpret_cast<const unsigned *>(stage + (r0 + i) * 128 + (((lane >> 2) ^ i) << 4) + (lane & 3) * 4);
#pragma unroll
                            for (int i = 0; i < 8; ++i) {
                                const long long o = o0 + static_cast<long long>(r0 + i) * q.cols;
                                if (q.out_f32) {
                                    float *const dst = static_cast<float *>(q.out) + o + lane;
                                    if (r0 + i < nr && lane < nc) {
                                        if (q.add) atomicAdd(dst, __uint_as_float(x[i]));
                                        else *dst = __uint_as_float(x[i]);
                                    }
                                } else {
                                    unsigned short *const row = static_cast<unsigned short *>(q.out) + o;
                                    const int odd = static_cast<int>(o & 1), at = 2 * lane + odd;
                                    const unsigned up = __shfl_down_sync(0xffffffffu, x[i], 1);
                                    const unsigned w = odd ? __funnelshift_r(x[i], up, 16) : x[i];
                                    if (r0 + i < nr) {
                                        if (at + 1 < nc) *reinterpret_cast<unsigned *>(row + at) = w;
                                        else if (at < nc) row[at] = static_cast<unsigned short>(w);
                                        if (odd && lane == 0) row[0] = static_cast<unsigned short>(x[i]);
                                    }
                                }
                            }
                        }
                        __syncwarp();
                    }
                }
            }
            tc_fence_before();
            warp_arrive(&pipe.acc_empty[slot]);
          }
        }
        if (lane == 0) bulk_wait_read_all();       // the staging block is read before the CTA goes
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, 512);
    }
}

bool fits_int(long long v) { return v > 0 && v < (1ll << 30); }

}  // namespace

// Steps of four MMAs per accumulator (see kMaxMmas): longer reductions of dW are split, longer ones of an fp32 dX (more than
// 8192 outputs) are cut into parts that follow one another, each added to the one before, so that the order of the sum is fixed.
// (A bf16 dX rounds far coarser than an accumulator does and is one part.)
constexpr long long kMaxSteps = kMaxMmas / 4;
// Clocks of a tile: its steps, whose cost is that of their hand-overs up to 128 columns and of their copies with 256, and its drain,
// which lies beside the next tile's steps where an accumulator holds a tile. plain: rows leave by ordinary stores. Fitted to 22
// layers timed in every form (64, 128, 256 columns, 128 or 256 rows, dW in one to eight parts): the form with the least estimate is
// within 0.8 % of the fastest on average, 6 % at worst.
double tile_clocks(int TN, int MA, long long steps, bool plain) {
    return steps * (TN < 256 ? 470.0 : MA == 2 ? 840.0 : 640.0) + (plain ? 20.0 * TN * MA : MA == 2 ? 5.0 * TN * MA : 300.0);
}

bool linear_tc_supported(long long B, long long N, long long K) { return fits_int(B) && fits_int(N) && fits_int(K); }

long long linear_pitch(long long cols) { return (cols + 7) / 8 * 8; }

// How the products of a layer are cut into tiles. Whether dW's reduction is split must be known before the statistics
// kernel runs (it clears dW on the side).
LinearPlan linear_plan(const dbp_ctx *ctx, long long B, long long N, long long K, int pieces, bool want_dw, bool want_dx) {
    LinearPlan pl;
    const long long dw_steps = ((B + 63) / 64) * pieces, dx_steps = ((N + 63) / 64) * pieces;
    // Split the weight gradient's reduction (into parts of at least four steps) where that shortens what the CTA with the most
    // work has, or when it is too long for one accumulator. dX is not split: its sums keep one order, so that the gradient handed
    // to the layer below is reproducible.
    auto span = [&](int tn, int ma, long long want) {                   // clocks of that CTA, as the kernel deals the tiles
        const long long rows = 128 * ma, nt = (K + tn - 1) / tn, per = (dw_steps + want - 1) / want, split = (dw_steps + per - 1) / per;
        long long n0 = want_dx ? (B + rows - 1) / rows * nt : 0, n1 = want_dw ? (N + rows - 1) / rows * nt * split : 0;
        double c0 = tile_clocks(tn, ma, dx_steps, pieces == 1 ? K % 8 != 0 : K % 4 != 0), c1 = tile_clocks(tn, ma, per, K % 4 != 0);
        if (!want_dx || (want_dw && per > dx_steps)) { std::swap(n0, n1); std::swap(c0, c1); }
        const long long G = n0 + n1 < ctx->sm_count ? n0 + n1 : ctx->sm_count, more = n0 % G;
        double a = (n0 / G + 1) * c0, b = n0 / G * c0;                  // CTAs with one more of the first product's tiles, and the others
        long long left = n1;
        if (more > 0) {
            const long long rounds = (left + G - more - 1) / (G - more), lead = static_cast<long long>(c0 / c1) < rounds ? static_cast<long long>(c0 / c1) : rounds;
            b += lead * c1;
            left -= lead * (G - more);
        }
        if (left > 0) {
            a += left / G * c1;
            b += (left + G - 1) / G * c1;
            if (left % G > G - more) a += c1;
        }
        // parts add into a dW that the statistics kernel clears
        const double parts = split > 1 ? static_cast<double>(N) * K * 4.0 / 2500.0 * (1.3 + 0.57 * split) : 0.0;
        return (more > 0 && a > b ? a : b) + parts + 3.0 * tn * ma;
    };
    const long long least = (dw_steps + kMaxSteps - 1) / kMaxSteps;
    // Columns, tile height and parts with the least work for the busiest CTA. Measured, us, before (columns by an estimate without
    // the dealing, one part unless SMs were idle, tiles of 128 rows dealt in turn) and now: bf16 1576 -> 66, B 4790: 57, 20 (split);
    // 360 -> 3208, B 6418: 119, 82 (256 rows, split); 560 -> 3476, B 848: 45, 28 (dealt); fp32 4048 -> 904, B 205: 36, 30 (dealt).
    // One or two parts add up to the same bits in whatever order they arrive (the cleared dW plus both), more do not: more are taken
    // only where they are a twentieth shorter, about as far as the estimate is off. Of 20000 layers of 16 to 8192 rows, 10 to 4096
    // outputs and 32 to 4096 inputs that costs the estimate 0.02 % on average (without the rule 1266 bf16 ones had more parts that
    // had one or two when only idle SMs were given parts, with it 1132).
    constexpr double kForOrder = 1.05;
    double shortest = 1e300, in_order = 1e300;
    long long want = least;
    LinearPlan ordered;
    long long ordered_want = least;
    for (int tn = 64; tn <= 256; tn *= 2) {
        if (tn > 64 && tn / 2 >= K) break;
        long long most = want_dw && dw_steps / 4 > least ? dw_steps / 4 : least;
        if (want_dw && K % 4 != 0) {
            // rows of dW that are no multiple of 16 bytes are added element by element: only on SMs that are idle otherwise (1072 x
            // 3806 x 1841 bf16: 102 us in one part, 236 in two)
            const long long nt = (K + tn - 1) / tn, idle = (ctx->sm_count - (want_dx ? (B + 127) / 128 * nt : 0)) / ((N + 127) / 128 * nt);
            if (most > idle) most = idle > least ? idle : least;
        }
        for (int ma = 1; ma <= (tn == 256 ? 2 : 1); ++ma)
            for (long long w = least; w <= most && w <= least + 16; ++w) {
                const double t = span(tn, ma, w);
                if (w <= 2 && t < in_order) { in_order = t; ordered.TN = tn; ordered.MA = ma; ordered_want = w; }
                if (t < shortest) { shortest = t; pl.TN = tn; pl.MA = ma; want = w; }
            }
    }
    if (in_order < kForOrder * shortest) { pl = ordered; want = ordered_want; }
    pl.dw_per_split = (dw_steps + want - 1) / want;
    pl.dw_split = (dw_steps + pl.dw_per_split - 1) / pl.dw_per_split;
    return pl;
}

namespace {
// dX from outputs [n0, n0 + len) of the reduction only
int launch_products(dbp_ctx *ctx, const LinearPlan &pl, const void *codes, const void *X, const void *W, int pieces,
                    long long x_pitch, long long w_pitch, const float *delta_p, long long B, long long N, long long K,
                    long long n0, long long len, float *dW, void *dX, bool dx_bf16, int *err_flag) {
    LinArgs p{};
    LinMaps maps;
    const long long q_pitch = linear_pitch(N);
    p.TN = pl.TN;
    p.MA = pl.MA;
    p.stage_bytes = p.MA * kABytesL + pl.TN / 64 * kPanelL;
    p.stages = kRingL / p.stage_bytes < kStagesL ? kRingL / p.stage_bytes : kStagesL;
    p.delta_p = delta_p;
    p.err_flag = err_flag;
    const int nt = static_cast<int>((K + pl.TN - 1) / pl.TN);
    // the product whose tiles take more reduction steps goes first
    const long long dx_steps = ((len + 63) / 64) * pieces;
    const bool dx_first = dX && (!dW || dx_steps >= pl.dw_per_split);
    auto fill = [&](bool is_dx) -> int {
        const int i = p.nprod++;
        LinProduct &q = p.pr[i];
        q.out = is_dx ? dX : dW;
        q.out_f32 = !(is_dx && dx_bf16);
        q.M = static_cast<int>(is_dx ? B : N);
        q.cols = static_cast<int>(K);
        q.a_kmajor = is_dx ? 1 : 0;
        const long long red = is_dx ? len : B;
        q.ks = static_cast<int>((red + 63) / 64);
        q.pieces = pieces;
        q.steps = q.ks * pieces;
        q.nsplit = is_dx ? 1 : static_cast<int>(pl.dw_split);
        q.per_split = is_dx ? q.steps : static_cast<int>(pl.dw_per_split);
        q.add = is_dx ? n0 > 0 : q.nsplit > 1;
        q.mt = (q.M + 128 * p.MA - 1) / (128 * p.MA);
        const long long tiles = static_cast<long long>(q.mt) * nt * q.nsplit;
        if (tiles + p.tiles >= (1ll << 30)) return DBP_EUNSUPPORTED;
        q.tiles = static_cast<int>(tiles);
        p.tiles += q.tiles;
        {
            const unsigned long long dims[2] = {static_cast<unsigned long long>(is_dx ? len : N), static_cast<unsigned long long>(B)};
            const unsigned long long str[1] = {static_cast<unsigned long long>(q_pitch) * 2};
            const unsigned box[2] = {64, is_dx ? 128u : 64u};
            if (!encode_map_bf16(&maps.a[i], static_cast<const unsigned short *>(codes) + (is_dx ? n0 : 0), 2, dims, str, box)) return fail_cuda("tensor map of the codes");
        }
        {
            const long long pitch = is_dx ? w_pitch : x_pitch;
            const unsigned long long dims[3] = {static_cast<unsigned long long>(K), static_cast<unsigned long long>(red),
                                                static_cast<unsigned long long>(pieces)};
            const unsigned long long str[2] = {static_cast<unsigned long long>(pitch) * 2,
                                               static_cast<unsigned long long>(pitch) * 2 * (is_dx ? N : B)};
            const unsigned box[3] = {64, 64, 1};
            const void *rows = is_dx ? static_cast<const unsigned short *>(W) + n0 * w_pitch : X;
            if (!encode_map_bf16(&maps.b[i], rows, 3, dims, str, box)) return fail_cuda("tensor map of an operand");
        }
        const int es = q.out_f32 ? 4 : 2;
        q.tma_out = (K * es) % 16 == 0 ? 1 : 0;
        if (q.tma_out) {
            const unsigned long long dims[2] = {static_cast<unsigned long long>(K), static_cast<unsigned long long>(q.M)};
            const unsigned long long str[1] = {static_cast<unsigned long long>(K) * es};
            const unsigned box[2] = {q.out_f32 ? 32u : 64u, 32};
            if (!(q.out_f32 ? encode_map_f32_sw128(&maps.out[i], q.out, 2, dims, str, box)
                            : encode_map_bf16(&maps.out[i], q.out, 2, dims, str, box)))
                return fail_cuda("tensor map of a product");
        }
        return DBP_OK;
    };
    int rc = DBP_OK;
    if (dX && dx_first) rc = fill(true);
    if (!rc && dW) rc = fill(false);
    if (!rc && dX && !dx_first) rc = fill(true);
    if (rc) return rc;
    const size_t smem = static_cast<size_t>(kRingL) + kEpiWarpsL * kOutBlock + 1024;
    const auto kern = p.MA == 2 ? linear_products_kernel<2> : linear_products_kernel<1>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
        return fail_cuda("shared memory size");
    const int grid = p.tiles < ctx->sm_count ? p.tiles : ctx->sm_count, more = p.pr[0].tiles % grid;
    if (p.nprod == 2 && more > 0) {
        auto clocks = [&](const LinProduct &q) { return tile_clocks(pl.TN, pl.MA, q.per_split, !q.tma_out); };
        const double ratio = clocks(p.pr[0]) / clocks(p.pr[1]), most = p.pr[1].tiles / (grid - more) + 1;
        p.lead = ratio < 1.0 ? 1 : static_cast<int>(ratio < most ? ratio : most);
    }
    return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(grid)), dim3(kThreadsL), smem, ctx->stream, maps, p));
}
}  // namespace

int launch_linear_products(dbp_ctx *ctx, const LinearPlan &pl, const void *codes, const void *X, const void *W, int pieces,
                           long long x_pitch, long long w_pitch, const float *delta_p, long long B, long long N, long long K,
                           float *dW, void *dX, bool dx_bf16, int *err_flag) {
    const long long most = dX && !dx_bf16 ? 64 * kMaxSteps : N;
    for (long long n0 = 0; n0 < N; n0 += most) {          // dW leaves with the first part of dX
        const long long len = N - n0 < most ? N - n0 : most;
        if (int rc = launch_products(ctx, pl, codes, X, W, pieces, x_pitch, w_pitch, delta_p, B, N, K, n0, len, n0 ? nullptr : dW, dX,
                                     dx_bf16, err_flag))
            return rc;
    }
    return DBP_OK;
}

}  // namespace dbp
