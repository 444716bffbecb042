// Input gradient of 3x3 convolutions (stride 1, pad 1) on small planes on the tensor cores (Eq. (qda)):
//   dX[b][ci][y][x] = Delta * sum_(co,ky,kx) q[b][co][y+1-ky][x+1-kx] * W[co][ci][ky][kx]
//
// The patches of tc3_tma_dx.cu carry a column of zeros per image row and a row of zeros per image, and multiply them: of an 8x8
// image's 81 columns 17 are thrown away, of a 2x2 image's nine 5, and every tap runs over all of them. Here a tile is ONE output row y
// of `nimg` images x 128 input channels. Its accumulator columns are numbered x * nimg + image, and a row of codes lies in shared
// memory in the same order, one 128-byte row of 64 output channels per (x', image), W copies of nimg rows each. A tap's
// columns are then a contiguous run: kx = 1 all of them, kx = 0 all but the last x (code rows from x' = 1 on), kx = 2 all but the
// first; kernel rows that leave the image do not exist. Nothing is computed and thrown away but images past the batch.
//
//   A = weights of one tap [64 co][128 ci]  (M = input channels, MN-major; from W re-laid as [tap][co][ci])
//   B = codes of one image row [W nimg][64 co]  (N = up to 256, K-major; a tap is a start row)
//   K = (64-channel block of co) x (input row) x (weight piece, low first) x (three taps), four MMAs of 16 channels each
//
// Bound by shared memory: per step (three taps of a piece) the copies write 48 KB of weights and the MMAs read them and
// 4 x 32 bytes per column of every tap; at N = 256 that is about 1500 clocks for 1408 of the tensor pipe (W = 8).
// The reduction over co may be split over a cluster of KS CTAs; partial sums are read through distributed shared memory 16
// bytes at a time and added in rank order (fixed: dX does not depend on timing).
// dX alone, us, this kernel against tc3_tma_dx.cu's, fp32, batch 128: 512 -> 512 at 4x4 30.6, 45.3; at 2x2 21.0, 29.2;
// 256 -> 512 at 4x4 23.6, 31.6; 128 -> 256 at 8x8 26.6, 33.2. VGG-16 layer set 680, 756.
//
// One tile per CTA (cluster). Warp 0 copies code rows, warp 1 weights, warp 2 issues the MMAs, warps 4-11 bring the
// accumulator to shared memory (over the operands, which nobody reads any more); then all warps add, transpose to image
// order and store. Every wait is bounded.
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace tc;

constexpr int kThreadsR = 12 * 32;
constexpr int kTapR = 64 * 128;                  // [64 co][64 ci] bf16
template <bool LEAN>
constexpr int kTapsR = LEAN ? 1 : 3;             // taps per weight slot (one hand-over)
template <bool LEAN>
constexpr int kSlotR = 2 * kTapsR<LEAN> * kTapR; // [panel of 64 ci][kx][64 co][64 ci]
constexpr int kMaxNWR = 4, kMaxNQR = 4;          // weight slots and code rows in flight, at most
constexpr int kMaxColsR = kRowsMaxCols;
constexpr int kTurnR = kMaxColsR + kMaxColsR / 16;   // words of a warp's row on its way from tile to image order

struct RowsDxP {
    const float *delta_p;
    void *dX;
    int B, Cin, H, W, HW;
    int nimg, N, N1;              // images per tile; accumulator columns W nimg, and those of the taps that lose one x
    int pitch;                    // words of a staged row: N rounded up to 32
    int groups, ci_tiles;
    int KS, ncb, pieces;
    int nw, nq;                   // weight slots, code rows in flight
    int es;                       // bytes per element of dX
    unsigned w_rcp;               // ceil(2^16 / W): i / W = i w_rcp >> 16 for i < 512, W <= 62
    int *err_flag;
    unsigned long long *stats;
};

struct PipeR {
    unsigned long long q_full[kMaxNQR], q_empty[kMaxNQR], w_full[kMaxNWR], w_empty[kMaxNWR], acc_full;
    unsigned tmem_base;
};

__device__ __forceinline__ void cluster_meet() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// LEAN: half an SM (shared memory, registers), a dW CTA beside it; weights tap by tap
template <bool LEAN>
__global__ void __launch_bounds__(kThreadsR, LEAN ? 2 : 1)
tc3_rows_dx_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_w, const RowsDxP p) {
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    constexpr int G = kTapsR<LEAN>, SLOT = kSlotR<LEAN>;
    const int q_bytes = p.N * 128;
    unsigned char *q_s = smem, *w_s = q_s + p.nq * q_bytes;
    float *stage = reinterpret_cast<float *>(smem);                  // [128 ci][pitch], 16-byte pieces swizzled by the row
    float *turn = stage + 128 * p.pitch;                             // a row per warp
    __shared__ PipeR pipe;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int KS = p.KS, rank = KS > 1 ? static_cast<int>(blockIdx.x) % KS : 0;      // consecutive CTAs are a cluster
    // tile: output rows with three input rows first
    int t = static_cast<int>(blockIdx.x) / KS;
    const int ci0 = t % p.ci_tiles * 128;
    t /= p.ci_tiles;
    const int b0 = t % p.groups * p.nimg, yi = t / p.groups;
    const int y = p.H == 1 ? 0 : yi < p.H - 2 ? yi + 1 : yi == p.H - 2 ? 0 : p.H - 1;
    const int y_lo = y > 0 ? y - 1 : 0, y_hi = y + 1 < p.H ? y + 1 : p.H - 1;
    const int c_lo = rank * p.ncb / KS, c_hi = (rank + 1) * p.ncb / KS;              // my 64-channel blocks of co

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxNQR; ++s) { mbar_init(&pipe.q_full[s], 1); mbar_init(&pipe.q_empty[s], 1); }
        for (int s = 0; s < kMaxNWR; ++s) { mbar_init(&pipe.w_full[s], 1); mbar_init(&pipe.w_empty[s], 1); }
        mbar_init(&pipe.acc_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_w);
    }
    if (warp == 2) tmem_alloc(&pipe.tmem_base, kMaxColsR);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem = pipe.tmem_base;
    if (KS > 1) cluster_meet();          // every CTA of the cluster is there before anybody reads its partial sums
    chain_wait();

    // taps of a kernel row in the order they are multiplied: kx = 1 first, which reaches every column
    auto kx_of = [](int g) { return g == 0 ? 1 : g == 1 ? 0 : 2; };
    const int hands = LEAN ? (p.W > 1 ? 3 : 1) : 1;                  // weight slots per step
    bool ok = true;
    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            unsigned parity = 1;                   // a fresh barrier passes a wait on the previous phase
            long long waited = 0;
            for (int c = c_lo; c < c_hi && ok; ++c)
                for (int yy = y_lo; yy <= y_hi; ++yy) {
                    ok = mbar_wait_timed(&pipe.q_empty[s], parity, p.err_flag, waited);
                    if (!ok) break;
                    mbar_expect_tx(&pipe.q_full[s], static_cast<unsigned>(q_bytes));
                    for (int x = 0; x < p.W; ++x)                    // images past the batch read as zero
                        tma_load_3d(q_s + s * q_bytes + x * p.nimg * 128, &map_q, c * 64, yy * p.W + x, b0, &pipe.q_full[s]);
                    if (++s == p.nq) { s = 0; parity ^= 1u; }
                }
            chain_release();
            report_wait(p.stats, 3, waited);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            int s = 0;
            unsigned parity = 1;
            long long waited = 0;
            for (int c = c_lo; c < c_hi && ok; ++c)
                for (int yy = y_lo; yy <= y_hi && ok; ++yy)
                    for (int piece = p.pieces - 1; piece >= 0 && ok; --piece)
                        for (int g = 0; g < hands; ++g) {
                            ok = mbar_wait_timed(&pipe.w_empty[s], parity, p.err_flag, waited);
                            if (!ok) break;
                            mbar_expect_tx(&pipe.w_full[s], SLOT);
                            for (int h = 0; h < 2; ++h)
                                tma_load_3d(w_s + s * SLOT + h * G * kTapR, &map_w, ci0 + 64 * h, c * 64,
                                            9 * piece + 3 * (y + 1 - yy) + (LEAN ? kx_of(g) : 0), &pipe.w_full[s]);
                            if (++s == p.nw) { s = 0; parity ^= 1u; }
                        }
            report_wait(p.stats, 4, waited);
        }
    } else if (warp == 2) {
        // the whole warp runs the loop (uniform control flow and operands); one elected lane issues
        const unsigned idesc = make_idesc(128, p.N, true, false), idesc1 = make_idesc(128, p.N1, true, false);
        const unsigned long long q_desc = make_desc(smem_u32(q_s), 16, 1024), w_desc = make_desc(smem_u32(w_s), G * kTapR, 1024);
        const unsigned one_x = static_cast<unsigned>(p.nimg * 8);    // the rows of one x, in 16-byte units
        int qs = 0, ws = 0;
        unsigned qpar = 0, wpar = 0, on = 0u;
        long long wq = 0, ww = 0;
        const long long born = clock64();
        for (int c = c_lo; c < c_hi && ok; ++c)
            for (int yy = y_lo; yy <= y_hi && ok; ++yy) {
                ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.q_full[qs], qpar, p.err_flag, wq));
                const unsigned long long bd = q_desc + static_cast<unsigned>(qs * (q_bytes >> 4));
                for (int hand = 0; hand < p.pieces * hands && ok; ++hand) {
                    ok = __all_sync(0xffffffffu, mbar_wait_timed(&pipe.w_full[ws], wpar, p.err_flag, ww));
                    if (!ok) break;
                    tc_fence_after();
                    const unsigned long long ad = w_desc + static_cast<unsigned>(ws * (SLOT >> 4));
                    const int g = LEAN ? hand % hands : 0;
                    if (elect_one()) {
                        // 16 co: 16 rows of A (2048 bytes), 32 bytes along a row of B
                        if (!LEAN || g == 0)
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_bf16(tmem, ad + (LEAN ? 0 : kTapR >> 4) + 128 * k, bd + 2 * k, idesc, k ? 1u : on);
                        if (LEAN ? g == 1 : p.N1 > 0)
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_bf16(tmem, ad + 128 * k, bd + one_x + 2 * k, idesc1, 1u);
                        if (LEAN ? g == 2 : p.N1 > 0)
#pragma unroll
                            for (int k = 0; k < 4; ++k) mma_bf16(tmem + p.nimg, ad + (LEAN ? 0 : 2 * (kTapR >> 4)) + 128 * k, bd + 2 * k, idesc1, 1u);
                        mma_commit(&pipe.w_empty[ws]);
                    }
                    on = 1u;
                    if (++ws == p.nw) { ws = 0; wpar ^= 1u; }
                }
                if (ok && elect_one()) mma_commit(&pipe.q_empty[qs]);
                if (++qs == p.nq) { qs = 0; qpar ^= 1u; }
            }
        if (ok && elect_one()) mma_commit(&pipe.acc_full);
        if (lane == 0) {
            report_wait(p.stats, 0, wq);
            report_wait(p.stats, 1, ww);
            report_wait(p.stats, 6, clock64() - born);
            report_wait(p.stats, 7, 1);
        }
    } else if (warp >= 4) {
        // TMEM lane = input channel, column = (x, image); two warps per lane quarter take turns at blocks of 32 columns
        const int q = warp & 3, row = q * 32 + lane;
        ok = __all_sync(0xffffffffu, mbar_wait(&pipe.acc_full, 0, p.err_flag));
        tc_fence_after();
        for (int c0 = (warp - 4) / 4 * 32; ok && c0 < p.N; c0 += 64) {
            unsigned v[32];
            tmem_ld32(tmem + (static_cast<unsigned>(q * 32) << 16) + c0, v);
            float4 *dst = reinterpret_cast<float4 *>(stage + row * p.pitch + c0);
#pragma unroll
            for (int h = 0; h < 8; ++h)
                dst[h ^ (row & 7)] = make_float4(__uint_as_float(v[4 * h]), __uint_as_float(v[4 * h + 1]), __uint_as_float(v[4 * h + 2]), __uint_as_float(v[4 * h + 3]));
        }
        tc_fence_before();
    }
    if (KS > 1) cluster_meet();
    else __syncthreads();
    // this CTA finishes 128 / KS channels, a warp a row at a time
    {
        const float delta = *p.delta_p;
        const int per = 128 / KS, nval = p.B - b0 < p.nimg ? p.B - b0 : p.nimg;
        float *const mine = turn + warp * kTurnR;
        unsigned base[8];
#pragma unroll
        for (int k = 0; k < 8; ++k)
            if (k < KS && KS > 1) asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(base[k]) : "r"(smem_u32(stage)), "r"(k));
        for (int r = warp; r < per; r += kThreadsR / 32) {
            const int row = rank * per + r, ci = ci0 + row;
            if (ci >= p.Cin) break;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const int c = half * 128 + lane * 4;
                if (c >= p.N) break;
                const int at = row * p.pitch + (c & ~31) + ((((c >> 2) ^ row) & 7) << 2);
                float4 s;
                if (KS == 1) {
                    s = *reinterpret_cast<const float4 *>(stage + at);
                } else {
                    float4 v[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k < KS)
                            asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                                         : "=f"(v[k].x), "=f"(v[k].y), "=f"(v[k].z), "=f"(v[k].w) : "r"(base[k] + 4 * at));
                    s = v[0];
#pragma unroll
                    for (int k = 1; k < 8; ++k)
                        if (k < KS) { s.x += v[k].x; s.y += v[k].y; s.z += v[k].z; s.w += v[k].w; }
                }
                // columns c .. c + 3 are four images of one x (nimg is a multiple of 16)
                const int x = c / p.nimg;
                int w = (c - x * p.nimg) * p.W + x;
                const float f[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
                for (int j = 0; j < 4; ++j, w += p.W) mine[w + (w >> 4)] = f[j] * delta;
            }
            __syncwarp();
            const long long o0 = (static_cast<long long>(b0) * p.Cin + ci) * p.HW + y * p.W;
            for (int i = lane; i < nval * p.W; i += 32) {
                const int img = static_cast<int>(static_cast<unsigned>(i) * p.w_rcp >> 16), x = i - img * p.W;
                const long long o = o0 + static_cast<long long>(img) * p.Cin * p.HW + x;
                const float f = mine[i + (i >> 4)];
                if (p.es == 4) static_cast<float *>(p.dX)[o] = f;
                else static_cast<__nv_bfloat16 *>(p.dX)[o] = __float2bfloat16_rn(f);
            }
            __syncwarp();
        }
    }
    if (KS > 1) cluster_meet();          // nobody leaves while its partial sums are still being read
    else __syncthreads();
    if (warp == 2) tmem_dealloc(tmem, kMaxColsR);
}

}  // namespace

// The cheapest tile and split by a count of clocks in the terms of launch_tc3_tma_dx's; < 0: not taken. Layers of more than 64 input
// channels (fewer put both weight pieces on the lanes there) and rows of up to 16 positions (16 images to a tile at least). An
// accumulator keeps to kMaxMmas: 36 MMAs per block of co and weight piece. (Nothing here depends on dX's type, so that a bf16 dX is
// the fp32 one rounded.)
double tc3_rows_plan(const dbp_ctx *ctx, const ConvShape &s, int pieces, int max_cols, RowsPlan *plan) {
    double best = -1.0;
    if (s.k != 3 || s.Cin <= 64 || s.W > 16 || s.H > 64 || ctx->phase_cin > 0) return best;
    const int sms = ctx->sm_count, ncb = static_cast<int>((s.Cout + 63) / 64), ci_tiles = static_cast<int>((s.Cin + 127) / 128);
    const int W = static_cast<int>(s.W), ky = s.H < 3 ? static_cast<int>(s.H) : 3;
    auto mma = [](double n) { return n <= 0 ? 0.0 : n / 2 > 32 + n / 4 ? n / 2 : 32 + n / 4; };
    for (int nimg = 16; nimg * W <= max_cols; nimg += 16) {
        if (nimg > 16 && nimg - 16 >= s.B) break;
        const int N = nimg * W, N1 = N - nimg;
        const long long groups = (s.B + nimg - 1) / nimg, tiles = groups * s.H * ci_tiles;
        if (tiles >= (1 << 20)) continue;
        for (int ks = 1; ks <= 8 && ks <= ncb; ks *= 2) {
            const int cbs = (ncb + ks - 1) / ks;
            if (cbs * 36 * pieces > kMaxMmas) continue;
            const long long ctas = tiles * ks;
            if (ks > 1 && ctas > (ks == 2 ? sms : ks == 4 ? sms * 7 / 8 : sms * 3 / 4)) continue;
            const long long waves = (ctas + sms - 1) / sms, active = ctas < sms ? ctas : sms;
            const double tensor = 4.0 * (mma(N) + 2 * mma(N1)), cols = N + 2.0 * N1, weights = kSlotR<false>, copied = weights + 128.0 * N / pieces;
            const double shared = (2.0 * weights + 128.0 * cols + 128.0 * N / pieces) / 128.0;
            const double rate = 6000.0 / active < 60.0 ? 6000.0 / active : 60.0;
            double step = tensor > shared ? tensor : shared;
            if (step < copied / rate) step = copied / rate;
            const double body = 1500.0 + cbs * ky * pieces * (step + 80.0);
            const double epi = 2500.0 + 128.0 * N * 4 / 32 + (ks > 1 ? 1000.0 + 128.0 * N * 4 / 25 : 0.0);
            const double cost = waves * (body + epi);
            if (best < 0 || cost < best) { best = cost; plan->nimg = nimg; plan->KS = ks; }
        }
    }
    return best;
}

// codes position-major [B][H W][q_pitch], weights re-laid in ctx->w_taps
int launch_tc3_rows_dx(dbp_ctx *ctx, const RowsPlan &plan, const void *codes_nhwc, int pieces, const float *delta_p, const ConvShape &s,
                       void *dX, bool dx_bf16, int *err_flag, bool *lean) {
    RowsDxP p{};
    p.delta_p = delta_p; p.dX = dX; p.err_flag = err_flag; p.stats = ctx->wait_stats;
    p.B = static_cast<int>(s.B); p.Cin = static_cast<int>(s.Cin); p.H = static_cast<int>(s.H); p.W = static_cast<int>(s.W);
    p.HW = p.H * p.W;
    p.nimg = plan.nimg; p.KS = plan.KS;
    p.N = p.nimg * p.W; p.N1 = p.N - p.nimg;
    p.pitch = (p.N + 31) / 32 * 32;
    p.groups = (p.B + p.nimg - 1) / p.nimg;
    p.ci_tiles = (p.Cin + 127) / 128;
    p.ncb = static_cast<int>((s.Cout + 63) / 64);
    p.pieces = pieces;
    p.es = dx_bf16 ? 2 : 4;
    p.w_rcp = (65536u + p.W - 1) / p.W;
    const unsigned ctas = static_cast<unsigned>(p.groups) * p.H * p.ci_tiles * p.KS;
    // half an SM's worth of it, when the caller can use the other half: tiles of up to kRowsLeanCols columns, one round of CTAs
    const bool small = lean != nullptr && p.N <= kRowsLeanCols && ctas <= static_cast<unsigned>(ctx->sm_count);
    if (lean != nullptr) *lean = small;
    // two code rows and as many weight slots as fit beside them; then more rows, as long as three (four small) slots are left
    const size_t row = static_cast<size_t>(p.N) * 128, budget = small ? kHalfSm - 1024 : 227 * 1024 - 2048, slot = small ? kSlotR<true> : kSlotR<false>;
    p.nq = 2;
    while (p.nq < kMaxNQR && (p.nq + 1) * row + (small ? 4 : 3) * slot <= budget) ++p.nq;
    const size_t rows = p.nq * row;
    p.nw = static_cast<int>((budget - rows) / slot);
    if (p.nw > kMaxNWR) p.nw = kMaxNWR;
    const size_t operands = rows + static_cast<size_t>(p.nw) * slot;
    const size_t sums = sizeof(float) * (128u * static_cast<size_t>(p.pitch) + kThreadsR / 32 * kTurnR);
    const size_t smem = (operands > sums ? operands : sums) + 1024;
    CUtensorMap map_q, map_w;
    const unsigned long long w_row = static_cast<unsigned long long>((s.Cin + 7) / 8 * 8) * 2, q_row = static_cast<unsigned long long>((s.Cout + 7) / 8 * 8) * 2;
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(s.Cout), static_cast<unsigned long long>(p.HW), static_cast<unsigned long long>(s.B)};
        const unsigned long long str[2] = {q_row, q_row * p.HW};
        const unsigned box[3] = {64, 1, static_cast<unsigned>(p.nimg)};
        if (!encode_map_bf16(&map_q, codes_nhwc, 3, dims, str, box)) return fail_cuda("tensor map of the code rows");
    }
    {
        const unsigned long long dims[3] = {static_cast<unsigned long long>(s.Cin), static_cast<unsigned long long>(s.Cout), 9ull * pieces};
        const unsigned long long str[2] = {w_row, w_row * s.Cout};
        const unsigned box[3] = {64, 64, small ? 1u : 3u};
        if (!encode_map_bf16(&map_w, ctx->w_taps.ptr, 3, dims, str, box)) return fail_cuda("tensor map of the weights");
    }
    const auto kern = small ? tc3_rows_dx_kernel<true> : tc3_rows_dx_kernel<false>;
    if (small) cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (allow_shared(kern) != cudaSuccess)
        return fail_cuda("shared memory size");
    if (p.KS > 1)
        return cuda_ok(launch_chained_cluster(kern, ctas, static_cast<unsigned>(p.KS), dim3(kThreadsR), smem, ctx->stream, map_q, map_w, p));
    return cuda_ok(launch_chained(kern, dim3(ctas), dim3(kThreadsR), smem, ctx->stream, map_q, map_w, p));
}

}  // namespace dbp
