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
// A CTA is persistent over output tiles of 128 rows x TN columns: warp 0 issues the copies, warp 1 the MMAs into
// one of two accumulators in tensor memory, warps 2-9 drain the other one (scale by Delta, convert, stage as
// 128-byte swizzled rows, one tiled store per 32-row block; rows whose pitch is no multiple of 16 bytes leave
// through plain stores). Weight-gradient tiles may be split along the reduction: the parts then add into a
// cleared dW through the copy engine.
// Large layers are bound by the tensor pipe (a step of 128 x 256 x 64 is 512 clocks of it against 48 KB of
// copies), small ones by the chain of reduction steps of one tile.
#include "tc_common.cuh"

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
    int mt;
    int tiles;                    // mt * column tiles * nsplit
};

struct LinArgs {
    LinProduct pr[2];             // the product with the longer tiles first
    int nprod, tiles, TN;
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

    // tile t -> product, first row and column, range of reduction steps
    struct Tile { int i, m0, n0, k0, k1; };
    auto tile_of = [&](int t) {
        Tile r;
        r.i = t < p.pr[0].tiles ? 0 : 1;
        const LinProduct &q = p.pr[r.i];
        if (r.i) t -= p.pr[0].tiles;
        const int s = t % q.nsplit;
        t /= q.nsplit;
        r.m0 = (t % q.mt) * 128;
        r.n0 = (t / q.mt) * p.TN;
        r.k0 = s * q.per_split;
        r.k1 = r.k0 + q.per_split < q.steps ? r.k0 + q.per_split : q.steps;
        return r;
    };

    if (warp == 0) {
        int s = 0;
        unsigned parity = 1;                     // a fresh barrier passes a wait on the previous phase
        bool ok = true;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x) {
            const Tile tl = tile_of(t);
            const LinProduct &q = p.pr[tl.i];
            const int left = (q.cols - tl.n0 + 63) >> 6;
            const int nb = left < p.TN / 64 ? left : p.TN / 64;      // 64-column panels that hold columns
            const unsigned tx = static_cast<unsigned>(kABytesL + nb * kPanelL);
            for (int k = tl.k0; k < tl.k1; ++k) {
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.empty[s], parity, p.err_flag));
                if (!ok) break;
                if (elect_one()) {
                    unsigned char *st = smem + s * stage_bytes;
                    // the low pieces first: the accumulator is still small when they are added
                    const int kp = k / q.ks, piece = q.pieces - 1 - kp, r0 = (k - kp * q.ks) * 64;
                    mbar_expect_tx(&pipe.full[s], tx);
                    if (q.a_kmajor) {
                        tma_load_2d(st, &maps.a[tl.i], r0, tl.m0, &pipe.full[s]);
                    } else {
                        tma_load_2d(st, &maps.a[tl.i], tl.m0, r0, &pipe.full[s]);
                        tma_load_2d(st + kPanelL, &maps.a[tl.i], tl.m0 + 64, r0, &pipe.full[s]);
                    }
                    st += kABytesL;
                    for (int i = 0; i < nb; ++i)
                        tma_load_3d(st + i * kPanelL, &maps.b[tl.i], tl.n0 + 64 * i, r0, piece, &pipe.full[s]);
                }
                if (++s == S) { s = 0; parity ^= 1u; }
            }
        }
    } else if (warp == 1) {
        const unsigned idesc_k = make_idesc(128, p.TN, false, true), idesc_mn = make_idesc(128, p.TN, true, true);
        int s = 0;
        unsigned parity = 0;
        bool ok = true;
        int it = 0;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x, ++it) {
            const Tile tl = tile_of(t);
            const bool kmaj = p.pr[tl.i].a_kmajor != 0;
            const int slot = it & 1;
            ok = __all_sync(0xffffffffu, mbar_wait(&pipe.acc_empty[slot], ((static_cast<unsigned>(it) >> 1) & 1u) ^ 1u, p.err_flag));
            if (!ok) break;
            tc_fence_after();
            const unsigned tmem_d = tmem_base + slot * kMaxNL;
            for (int k = tl.k0; k < tl.k1; ++k) {
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.full[s], parity, p.err_flag));
                if (!ok) break;
                tc_fence_after();
                const unsigned a_addr = smem_u32(smem + s * stage_bytes);
                const unsigned long long bd = make_desc(a_addr + kABytesL, kPanelL, 1024);
                if (elect_one()) {
                    if (kmaj) {
                        const unsigned long long ad = make_desc(a_addr, 16, 1024);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)       // 16 along the rows of A = 32 bytes
                            mma_bf16(tmem_d, ad + 2 * kk, bd + 128 * kk, idesc_k, (k > tl.k0 || kk > 0) ? 1u : 0u);
                    } else {
                        const unsigned long long ad = make_desc(a_addr, kPanelL, 1024);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)       // 16 rows of A = 2048 bytes
                            mma_bf16(tmem_d, ad + 128 * kk, bd + 128 * kk, idesc_mn, (k > tl.k0 || kk > 0) ? 1u : 0u);
                    }
                    mma_commit(&pipe.empty[s]);
                }
                if (++s == S) { s = 0; parity ^= 1u; }
            }
            if (ok && elect_one()) mma_commit(&pipe.acc_full[slot]);
        }
    } else {
        // epilogue: TMEM lane = output row, column = output column; two warps per lane quarter take turns at the
        // blocks of 32 fp32 or 64 bf16 columns (128 bytes of a row)
        const int q4 = warp & 3, part = (warp - 2) >> 2;
        unsigned char *stage = smem + kRingL + (warp - 2) * kOutBlock;
        const float delta = *p.delta_p;
        bool ok = true;
        int it = 0;
        for (int t = blockIdx.x; t < p.tiles && ok; t += gridDim.x, ++it) {
            const Tile tl = tile_of(t);
            const LinProduct &q = p.pr[tl.i];
            const int slot = it & 1;
            ok = mbar_wait(&pipe.acc_full[slot], (static_cast<unsigned>(it) >> 1) & 1u, p.err_flag);
            if (!ok) break;
            tc_fence_after();
            const int row_w = tl.m0 + q4 * 32;                     // first output row of this warp
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
                        const int nr = q.M - row_w < 32 ? q.M - row_w : 32;
                        const int nc = ncol - c < bw ? ncol - c : bw;
                        const long long o0 = static_cast<long long>(row_w) * q.cols + tl.n0 + c;
                        for (int r = 0; r < nr; ++r) {
                            const long long o = o0 + static_cast<long long>(r) * q.cols;
                            if (q.out_f32) {
                                const float f = *reinterpret_cast<const float *>(stage + r * 128 + (((lane >> 2) ^ (r & 7)) << 4) + (lane & 3) * 4);
                                if (lane < nc) {
                                    if (q.add) atomicAdd(static_cast<float *>(q.out) + o + lane, f);
                                    else static_cast<float *>(q.out)[o + lane] = f;
                                }
                            } else {
                                for (int i = lane; i < nc; i += 32)
                                    static_cast<unsigned short *>(q.out)[o + i] =
                                        *reinterpret_cast<const unsigned short *>(stage + r * 128 + (((i >> 3) ^ (r & 7)) << 4) + (i & 7) * 2);
                            }
                        }
                        __syncwarp();
                    }
                }
            }
            tc_fence_before();
            warp_arrive(&pipe.acc_empty[slot]);
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

bool linear_tc_supported(long long B, long long N, long long K) { return fits_int(B) && fits_int(N) && fits_int(K); }

long long linear_pitch(long long cols) { return (cols + 7) / 8 * 8; }

// How the products of a layer are cut into tiles. Whether dW's reduction is split must be known before the statistics
// kernel runs (it clears dW on the side).
LinearPlan linear_plan(const dbp_ctx *ctx, long long B, long long N, long long K, int pieces, bool want_dw, bool want_dx) {
    LinearPlan pl;
    const long long dw_steps = ((B + 63) / 64) * pieces, dx_steps = ((N + 63) / 64) * pieces;
    // The shortest makespan of tiles of 256, 128 or 64 columns: a step of a 128 x 256 tile is 512 clocks of the tensor
    // pipe, narrower ones are bound by their copies and hand-overs (about 420 and 400 clocks); a tile ends with a drain of
    // about 4 clocks a column. Measured, us, for 64 / 128 / 256 columns: bf16 1024 -> 4096, B 4096: 213 / 144 / 96; fp32
    // 1024 -> 100, B 1024: 25 / 15.2 / 16.2; bf16 512 -> 512, B 512: 11.9 / 12.3 / 14.0.
    double best = 1e300;
    for (int tn = 64; tn <= 256; tn *= 2) {
        if (tn > 64 && tn / 2 >= K) break;
        const double step = tn == 256 ? 520.0 : tn == 128 ? 420.0 : 400.0, drain = 4.0 * tn + 500.0;
        const double nt = static_cast<double>((K + tn - 1) / tn);
        const double dx = want_dx ? dx_steps * step + drain : 0.0, dw = want_dw ? dw_steps * step + drain : 0.0;
        const double all = nt * ((B + 127) / 128) * dx + nt * ((N + 127) / 128) * dw;
        double longest = dx;                                            // (long dW reductions are split)
        if (longest < all / ctx->sm_count) longest = all / ctx->sm_count;
        if (longest < best) { best = longest; pl.TN = tn; }
    }
    const long long nt = (K + pl.TN - 1) / pl.TN;
    const long long dx_tiles = want_dx ? ((B + 127) / 128) * nt : 0;
    const long long dw_tiles = want_dw ? ((N + 127) / 128) * nt : 0;
    // Split the weight gradient's reduction when its tiles leave SMs idle (parts of at least four steps) and when it
    // is too long for one accumulator. dX is not split: its sums keep one order, so that the gradient handed to the
    // layer below is reproducible.
    const long long idle = ctx->sm_count - dx_tiles;
    long long want = 1;
    if (want_dw && dw_tiles < idle) {
        want = idle / dw_tiles;
        if (want > dw_steps / 4) want = dw_steps / 4;
        if (want < 1) want = 1;
    }
    if (want < (dw_steps + kMaxSteps - 1) / kMaxSteps) want = (dw_steps + kMaxSteps - 1) / kMaxSteps;
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
    p.stage_bytes = kABytesL + pl.TN / 64 * kPanelL;
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
        q.mt = (q.M + 127) / 128;
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
    if (cudaFuncSetAttribute(linear_products_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
        return fail_cuda("shared memory size");
    const int grid = p.tiles < ctx->sm_count ? p.tiles : ctx->sm_count;
    return cuda_ok(launch_chained(linear_products_kernel, dim3(static_cast<unsigned>(grid)), dim3(kThreadsL), smem, ctx->stream, maps, p));
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
