// Quantization and both products of a thin bf16 1x1 layer in one kernel (Eqs. (nsd), (qda), (qdw)):
//   q = floor(delta / Delta + u),   dX[b, ci, p] = Delta sum_co W[co, ci] q[b, co, p],   dW[co, ci] = Delta sum_{b, p} q[b, co, p] X[b, ci, p]
//
// A 64-channel x 64-position tile of codes in shared memory, one 128-byte swizzled row per output channel, is a valid
// operand of both products: for dX its rows are the reduction (MN-major, N = positions), for dW its rows are the output
// channels (K-major, M = channels). So where the whole of W and all of dW fit one CTA (tensor memory: dW accumulators of the
// whole layer beside two dX accumulators), delta is read once after the statistics, the codes never leave the SM, and
// quantization (instruction issue), products (tensor pipe) and the copies of X and dX (memory) run beside one another.
// Before: the quantizer wrote bf16 codes that two kernels read again. 64 -> 256 at 56x56, batch 64 (51 M gradient elements):
// 119 -> 72 us for the whole call, of which this kernel 53.
//
// A CTA is persistent over tiles of NCH chunks of 64 positions. Warp 0 copies delta: a stage is ROWS output channels of the
// tile, and its buffer holds delta first and the codes after, row by row in the same swizzled place, so that a quantizer
// thread has no addresses to make and no edges to look at (the copy engine reads zeros outside the tensor) and every stage of
// the ring is in flight. Warp 1 issues the MMAs, warps 2-5 drain the dX accumulators (and dW at the end, added into the
// cleared dW by the copy engine), warps 6-21 quantize, warp 22 copies W (once) and X. Where the vectors came to the
// quantizer's registers by plain loads instead, 64 bytes a thread ahead, the call above took 84 us against 72: the kernel
// executed 27 instructions an element against 21.
// Sixteen quantizer warps, and four that drain, rather than eight of each: 84 against 139 us (of that form), because two
// warps per scheduler do not hide the latencies of the dither's multiplications. The step size is added up from the
// statistics kernel's partial sums by every CTA (step_of).
// Bound by the quantizer's instructions: 15 of the 21 are the decision, which takes 22 clocks an element and scheduler (30 us
// of this kernel's 53); copies, MMAs and stores alone, with the codes left out, take 37 (by themselves, cold).
#include "nsd_common.cuh"
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace tc;
using namespace nsd;

constexpr int kQWarps = 16, kEWarps = 4;
constexpr int kXWarp = 2 + kEWarps + kQWarps;    // copies W and X
constexpr int kThreadsF = 32 * (kXWarp + 1);
constexpr int kPanelF = 128 * 128;               // [128 co][64 positions] bf16
constexpr int kMaxStages = 6;
constexpr int kOutF = 32 * 128;                  // one epilogue warp's staging block

struct Fused1P {
    const __nv_bfloat16 *delta;
    unsigned long long seed;
    DeviceState *st;
    int Cin, Cout, HW, B;
    int cpi, nchunks, ntiles;     // 64-position chunks per image, in all; tiles
    int nco;                      // stages per tile
    int w_panels, w_rows;         // resident W: 64-channel panels of ci, rows (co) per panel
    int NT, NTp;                  // dW columns, rounded to 16 and to 32
    int MA;                       // 128-channel accumulators of dX per tile
    int stages;
    // the dither's counter: of the pair of elements 2 i, 2 i + 1: seed + (i + 1) gamma. A tile's chunks lie step_c chunks (within
    // an image) and tile_z of the counter (from behind the last stage) before those of the CTA's tile before it, and wrap_z
    // after that where the step passes the first chunk of an image; stage_z: a stage's channels, row64_z: 64 channels
    int step_c;
    unsigned long long tile_z, wrap_z, stage_z, row64_z;
    int *err_flag;
};

struct PipeF {
    unsigned long long d_full[kMaxStages], q_full[kMaxStages], q_empty[kMaxStages], x_full[2], x_empty[2], w_full, acc_full[2], acc_empty[2], dw_full;
    unsigned tmem_base;
};

template <int ROWS, int NCH>
__global__ void __launch_bounds__(kThreadsF, 1)
fused1x1_kernel(const __grid_constant__ CUtensorMap map_d, const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_x,
                const __grid_constant__ CUtensorMap map_dx, const __grid_constant__ CUtensorMap map_dw,
                const StepSource step, const Fused1P p) {
    constexpr int NV = ROWS * NCH * 8 / (32 * kQWarps);              // vectors per quantizer thread and stage
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *smem = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int w_bytes = p.w_panels * p.w_rows * 128, x_bytes = NCH * p.NT * 128;
    unsigned char *w_s = smem, *x_s = w_s + w_bytes, *q_s = x_s + 2 * x_bytes, *out_s = q_s + p.stages * NCH * kPanelF;
    __shared__ PipeF pipe;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = p.stages;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kMaxStages; ++s) { mbar_init(&pipe.d_full[s], 1); mbar_init(&pipe.q_full[s], kQWarps); mbar_init(&pipe.q_empty[s], 1); }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&pipe.x_full[s], 1); mbar_init(&pipe.x_empty[s], 1);
            mbar_init(&pipe.acc_full[s], 1); mbar_init(&pipe.acc_empty[s], kEWarps);
        }
        mbar_init(&pipe.w_full, 1);
        mbar_init(&pipe.dw_full, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tma_prefetch_desc(&map_d);
        tma_prefetch_desc(&map_w);
        tma_prefetch_desc(&map_x);
        tma_prefetch_desc(&map_dx);
        tma_prefetch_desc(&map_dw);
    }
    if (warp == 1) tmem_alloc(&pipe.tmem_base, 512);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const unsigned tmem_base = pipe.tmem_base, tmem_dx = tmem_base + p.nco * p.NTp;

    // tile i of this CTA: tiles are taken from the last one down (the end of delta is what the statistics left in the L2)
    struct Chunk { int b, p0; };
    auto tile_of = [&](int i) { return p.ntiles - 1 - static_cast<int>(blockIdx.x) - i * static_cast<int>(gridDim.x); };
    auto chunk_of = [&](int t, int j) {
        const int g = t * NCH + j, b = g / p.cpi;
        return Chunk{b, (g - b * p.cpi) * 64};
    };
    const int my_tiles = (p.ntiles - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);

    // delta, X and W are inputs of the call: their first tiles are on their way while the statistics kernel runs (it lets
    // this kernel start when all of its blocks have seen everything before them complete)
    // delta comes as the codes will lie: a stage's buffer holds it first
    const int total = my_tiles * p.nco;
    auto load_d = [&](int n, int s) {
        const int i = n / p.nco, co = (n - i * p.nco) * ROWS, t = tile_of(i);
        mbar_expect_tx(&pipe.d_full[s], NCH * ROWS * 128);
        for (int j = 0; j < NCH; ++j) {          // what lies outside the tensor reads as zero
            const Chunk c = chunk_of(t, j);
            tma_load_3d(q_s + s * NCH * kPanelF + j * kPanelF, &map_d, c.p0, co, c.b, &pipe.d_full[s]);
        }
    };
    auto load_x = [&](int i) {
        const int t = tile_of(i), s = i & 1;
        const int nch = p.nchunks - t * NCH < NCH ? p.nchunks - t * NCH : NCH;
        mbar_expect_tx(&pipe.x_full[s], static_cast<unsigned>(nch * p.NT * 128));
        for (int j = 0; j < nch; ++j) {
            const Chunk c = chunk_of(t, j);
            tma_load_3d(x_s + s * x_bytes + j * p.NT * 128, &map_x, c.p0, 0, c.b, &pipe.x_full[s]);
        }
    };
    if (threadIdx.x == 0) {
        for (int n = 0; n < S && n < total; ++n) load_d(n, n);
    } else if (threadIdx.x == 32 * kXWarp) {
        mbar_expect_tx(&pipe.w_full, static_cast<unsigned>(w_bytes));
        for (int h = 0; h < p.w_panels; ++h)
            for (int r = 0; r < p.w_rows; r += 64)
                tma_load_2d(w_s + (h * p.w_rows + r) * 128, &map_w, 64 * h, r, &pipe.w_full);
        load_x(0);
        if (my_tiles > 1) load_x(1);
    }
    const StepSource from = step_ahead(step);
    chain_wait();
    const float delta = step_of<kThreadsF>(from, p.st);

    if (warp == 0) {
        if (lane == 0) {
            int s = 0;
            unsigned par = 0;                                        // stage n again once the MMAs of stage n - S have read it
            int n = S;
            for (; n < total; ++n) {
                if (!mbar_wait(&pipe.q_empty[s], par, p.err_flag)) break;
                load_d(n, s);
                if (++s == S) { s = 0; par ^= 1u; }
            }
            if (n < total)                                           // given up: no copy may outlive the CTA
                for (int k = 0; k < S; ++k) mbar_wait(&pipe.d_full[k], ((n - k + S - 1) / S - 1) & 1, p.err_flag);
            chain_release();
        }
    } else if (warp == kXWarp) {
        if (lane == 0)
            for (int i = 2; i < my_tiles; ++i) {
                if (!mbar_wait(&pipe.x_empty[i & 1], ((i >> 1) & 1) ^ 1, p.err_flag)) {
                    for (int k = i - 2; k < i; ++k) mbar_wait(&pipe.x_full[k & 1], (k >> 1) & 1, p.err_flag);
                    break;
                }
                load_x(i);
            }
    } else if (warp == 1) {
        // the whole warp runs the loop (uniform control flow and operands); one elected lane issues
        const unsigned idesc_dx = make_idesc(128, 64 * NCH, true, true), idesc_dw = make_idesc(128, p.NT, false, false);
        const unsigned long long w_desc = make_desc(smem_u32(w_s), p.w_panels > 1 ? p.w_rows * 128 : 0, 1024);
        const unsigned w_ma = static_cast<unsigned>(2 * p.w_rows * 128) >> 4;        // two panels further: the next 128 channels
        int s = 0, n = 0;
        unsigned par = 0;
        bool ok = __all_sync(0xffffffffu, mbar_wait(&pipe.w_full, 0, p.err_flag));
        for (int i = 0; i < my_tiles && ok; ++i) {
            const int slot = i & 1, t = tile_of(i);
            ok = __all_sync(0xffffffffu, mbar_wait(&pipe.acc_empty[slot], ((i >> 1) & 1) ^ 1, p.err_flag)) &&
                 __all_sync(0xffffffffu, mbar_wait(&pipe.x_full[slot], (i >> 1) & 1, p.err_flag));
            if (!ok) break;
            const unsigned d_dx = tmem_dx + slot * p.MA * 64 * NCH;
            const unsigned long long x_desc = make_desc(smem_u32(x_s + slot * x_bytes), 16, 1024);
            int nk[NCH];                                             // 16-position slices that hold positions
#pragma unroll
            for (int j = 0; j < NCH; ++j) {
                const Chunk c = chunk_of(t, j);
                const int left = p.HW - c.p0;
                nk[j] = c.b >= p.B ? 0 : left >= 64 ? 4 : (left + 15) >> 4;
            }
            for (int cb = 0; cb < p.nco && ok; ++cb, ++n) {
                ok = __all_sync(0xffffffffu, mbar_wait(&pipe.q_full[s], par, p.err_flag));
                if (!ok) break;
                tc_fence_after();
                const unsigned q_addr = smem_u32(q_s + s * NCH * kPanelF);
                const unsigned long long qb = make_desc(q_addr, kPanelF, 1024), qa = make_desc(q_addr, 16, 1024);
                const unsigned long long wd = w_desc + static_cast<unsigned>(cb * ROWS * 128 >> 4);
                const int left = p.Cout - cb * ROWS, kr = ((left < ROWS ? left : ROWS) + 15) >> 4;
                if (elect_one()) {
                    for (int a = 0; a < p.MA; ++a) {
                        const unsigned long long ad = wd + static_cast<unsigned>(a) * w_ma;
                        if (kr == ROWS / 16) {
#pragma unroll
                            for (int k = 0; k < ROWS / 16; ++k)      // 16 rows = 2048 bytes
                                mma_bf16(d_dx + a * 64 * NCH, ad + 128 * k, qb + 128 * k, idesc_dx, (cb > 0 || k > 0) ? 1u : 0u);
                        } else {
                            for (int k = 0; k < kr; ++k)
                                mma_bf16(d_dx + a * 64 * NCH, ad + 128 * k, qb + 128 * k, idesc_dx, (cb > 0 || k > 0) ? 1u : 0u);
                        }
                    }
#pragma unroll
                    for (int j = 0; j < NCH; ++j) {
                        const unsigned long long ad = qa + j * (kPanelF >> 4), bd = x_desc + static_cast<unsigned>(j * p.NT * 128 >> 4);
                        for (int k = 0; k < nk[j]; ++k)              // 16 positions = 32 bytes
                            mma_bf16(tmem_base + cb * p.NTp, ad + 2 * k, bd + 2 * k, idesc_dw, (i > 0 || j > 0 || k > 0) ? 1u : 0u);
                    }
                    mma_commit(&pipe.q_empty[s]);
                }
                if (++s == S) { s = 0; par ^= 1u; }
            }
            if (ok && elect_one()) {
                mma_commit(&pipe.acc_full[slot]);
                mma_commit(&pipe.x_empty[slot]);
            }
        }
        if (ok && elect_one()) mma_commit(&pipe.dw_full);
    } else if (warp < 2 + kEWarps) {
        // epilogue: TMEM lane = input channel, column = position; two warps per lane quarter share a tile's blocks of
        // 32 channels x 64 positions: scaled, rounded, staged as swizzled 128-byte rows, one tiled store each
        const int q = warp & 3, part = (warp - 2) >> 2, parts = kEWarps / 4;
        unsigned char *stage = out_s + (warp - 2) * kOutF;
        bool ok = true;
        for (int i = 0; i < my_tiles && ok; ++i) {
            const int slot = i & 1, t = tile_of(i);
            ok = mbar_wait(&pipe.acc_full[slot], (i >> 1) & 1, p.err_flag);
            if (!ok) break;
            tc_fence_after();
            for (int k = part; k < p.MA * NCH; k += parts) {
                const int a = k / NCH, j = k - a * NCH, ci_w = a * 128 + q * 32;
                const Chunk c = chunk_of(t, j);
                if (c.b >= p.B || ci_w >= p.Cin) continue;           // warp-uniform
                unsigned v0[32], v1[32];
                const unsigned taddr = tmem_dx + (static_cast<unsigned>(q * 32) << 16) + (slot * p.MA + a) * 64 * NCH + j * 64;
                tmem_ld32(taddr, v0);
                tmem_ld32(taddr + 32, v1);
                if (lane == 0) bulk_wait_read_all();                 // the block's previous store has been read
                __syncwarp();
#pragma unroll
                for (int h = 0; h < 8; ++h) {
                    unsigned w[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const int x = 8 * (h & 3) + 2 * e;
                        const __nv_bfloat162 b2 = __floats2bfloat162_rn(__uint_as_float(h < 4 ? v0[x] : v1[x]) * delta,
                                                                        __uint_as_float(h < 4 ? v0[x + 1] : v1[x + 1]) * delta);
                        w[e] = *reinterpret_cast<const unsigned *>(&b2);
                    }
                    *reinterpret_cast<uint4 *>(stage + lane * 128 + ((h ^ (lane & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
                fence_async_proxy();
                __syncwarp();
                if (lane == 0) {                                     // what lies outside the tensor is skipped
                    tma_store_3d(&map_dx, c.p0, ci_w, c.b, stage);
                    bulk_commit();
                }
            }
            tc_fence_before();
            warp_arrive(&pipe.acc_empty[slot]);
        }
        // dW: TMEM lane = output channel (row of a stage), column = input channel
        if (ok && mbar_wait(&pipe.dw_full, 0, p.err_flag)) {
            tc_fence_after();
            const int per = (p.NT + 31) >> 5;
            for (int k = part; k < p.nco * per; k += parts) {
                const int cb = k / per, c0 = (k - cb * per) * 32, co_w = cb * ROWS + q * 32;
                if (q * 32 >= ROWS || co_w >= p.Cout) continue;      // warp-uniform; a stage of 64 rows fills half the lanes
                unsigned v[32];
                tmem_ld32(tmem_base + (static_cast<unsigned>(q * 32) << 16) + cb * p.NTp + c0, v);
                if (lane == 0) bulk_wait_read_all();
                __syncwarp();
#pragma unroll
                for (int h = 0; h < 8; ++h)
                    *reinterpret_cast<float4 *>(stage + lane * 128 + ((h ^ (lane & 7)) << 4)) =
                        make_float4(__uint_as_float(v[4 * h]) * delta, __uint_as_float(v[4 * h + 1]) * delta,
                                    __uint_as_float(v[4 * h + 2]) * delta, __uint_as_float(v[4 * h + 3]) * delta);
                fence_async_proxy();
                __syncwarp();
                if (lane == 0) {
                    tma_reduce_add_2d(&map_dw, c0, co_w, stage);
                    bulk_commit();
                }
            }
        }
        if (lane == 0) bulk_wait_read_all();
    } else {
        const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;          // Delta = 0: every code 0
        unsigned sat = 0, nnz = 0, nz2 = 0;
        int s = 0;
        unsigned par = 0;
        // A thread takes the same eight positions of rows qrow, qrow + 64 of every chunk of a stage, in place
        constexpr int RPC = NV / NCH;                                // its rows of a chunk
        const int qt = threadIdx.x - 32 * (2 + kEWarps), c8 = (qt & 7) * 8, qrow = qt >> 3;
        unsigned char *const mine = q_s + qrow * 128 + (((qt & 7) ^ (qrow & 7)) << 4);      // (row & 7 is the same for all its rows)
        int fc[NCH];                                                 // per chunk: its number in its image
        unsigned long long z[NCH];                                   // and the counter of the first row's first pair
#pragma unroll
        for (int j = 0; j < NCH; ++j) {
            const Chunk c = chunk_of(tile_of(0), j);
            fc[j] = c.p0 >> 6;
            z[j] = counter_of((static_cast<long long>(c.b) * p.Cout + qrow) * p.HW + c.p0 + c8, p.seed);
        }
        int left = p.nco;                                            // stages of the tile
        for (int n = 0; n < total; ++n) {
            if (!__all_sync(0xffffffffu, mbar_wait(&pipe.d_full[s], par, p.err_flag))) break;
            unsigned char *dst = mine + s * NCH * kPanelF;
            uint4 raw[NV];
            unsigned top = 0u;
            const unsigned before = nz2;
#pragma unroll
            for (int k = 0; k < NV; ++k) raw[k] = *reinterpret_cast<const uint4 *>(dst + k / RPC * kPanelF + k % RPC * 64 * 128);
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float x[8];
                unsigned long long u[4];
                unsigned h[4];
                Vec<__nv_bfloat16>::values(raw[k], x);
                dithers_at<8>(z[k / RPC] + k % RPC * p.row64_z, u);
                quick_codes<8>(x, u, inv, h, top);                   // outside the tensor x is 0: code 0
                count_pairs<8>(h, nz2);
                *reinterpret_cast<uint4 *>(dst + k / RPC * kPanelF + k % RPC * 64 * 128) = make_uint4(h[0], h[1], h[2], h[3]);
            }
            if (needs_care(top)) {                                   // rare: clip, count, NaN; from delta in memory again
                const int t = tile_of(n / p.nco), co0 = n % p.nco * ROWS + qrow;
                nz2 = before;
#pragma unroll 1
                for (int k = 0; k < NV; ++k) {
                    const Chunk c = chunk_of(t, k / RPC);
                    const int co = co0 + k % RPC * 64;
                    uint4 q = make_uint4(0u, 0u, 0u, 0u);
                    const long long e = (static_cast<long long>(c.b) * p.Cout + co) * p.HW + c.p0 + c8;
                    if (c.b < p.B && c.p0 + c8 < p.HW && co < p.Cout) q = __ldg(reinterpret_cast<const uint4 *>(p.delta + e));
                    float x[8];
                    unsigned long long u[4];
                    unsigned h[4], m[8];
                    Vec<__nv_bfloat16>::values(q, x);
                    dithers_of<8>(e, p.seed, u);
                    careful_codes<8>(x, u, inv, h, m, sat);
                    count_pairs<8>(h, nz2);
                    *reinterpret_cast<uint4 *>(dst + k / RPC * kPanelF + k % RPC * 64 * 128) = make_uint4(h[0], h[1], h[2], h[3]);
                }
            }
            fence_async_proxy();
            warp_arrive(&pipe.q_full[s]);
            if (++s == S) { s = 0; par ^= 1u; }
            if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
#pragma unroll
            for (int j = 0; j < NCH; ++j) z[j] += p.stage_z;
            if (--left == 0) {                                       // the next tile
                left = p.nco;
#pragma unroll
                for (int j = 0; j < NCH; ++j) {
                    fc[j] -= p.step_c;
                    z[j] -= p.tile_z;
                    if (fc[j] < 0) { fc[j] += p.cpi; z[j] += p.wrap_z; }
                }
            }
        }
        nnz = __reduce_add_sync(kFull, nnz + pairs_total(nz2));
        sat = __reduce_add_sync(kFull, delta > 0.f ? sat : 0u);
        if (lane == 0) {
            if (nnz) atomicAdd(&p.st->nnz, static_cast<unsigned long long>(nnz));
            if (sat) atomicAdd(&p.st->saturated, static_cast<unsigned long long>(sat));
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        __syncwarp();
        tmem_dealloc(tmem_base, 512);
    }
}

// Tiles, accumulators and buffers of a layer; false where they do not fit or the tiles are too few to fill the GPU evenly.
bool plan_fused1x1(const ConvShape &s, int sms, Fused1P &p, int &rows, int &nch, size_t &smem) {
    const long long HW = s.H * s.W;
    if (s.k != 1 || HW % 8 != 0 || HW < 64 || s.Cin % 8 != 0 || s.Cin > 256 || s.Cout > 512 || s.B * s.Cout * HW >= (1ll << 40)) return false;
    p.Cin = static_cast<int>(s.Cin); p.Cout = static_cast<int>(s.Cout); p.B = static_cast<int>(s.B); p.HW = static_cast<int>(HW);
    p.cpi = static_cast<int>((HW + 63) / 64);
    if (s.B * p.cpi >= (1ll << 30)) return false;
    p.nchunks = p.B * p.cpi;
    rows = p.Cout <= 64 ? 64 : 128;
    p.nco = (p.Cout + rows - 1) / rows;
    p.NT = (p.Cin + 15) / 16 * 16;
    p.NTp = (p.NT + 31) / 32 * 32;
    p.MA = (p.Cin + 127) / 128;
    p.w_panels = (p.Cin + 63) / 64;
    p.w_rows = (p.Cout + 63) / 64 * 64;
    for (nch = 2; nch >= 1; --nch) {
        if (p.nco * p.NTp + 2 * p.MA * 64 * nch > 512) continue;
        p.ntiles = (p.nchunks + nch - 1) / nch;
        if (p.ntiles < 2 * sms) continue;
        // (the last stage of dX reads whole 128-row panels: a panel is allocated whole even where its rows are 64)
        const size_t fixed = static_cast<size_t>(p.w_panels) * p.w_rows * 128 + 2 * static_cast<size_t>(nch) * p.NT * 128 + kEWarps * kOutF + 1024;
        const size_t budget = 227 * 1024 - 2048, stage = static_cast<size_t>(nch) * kPanelF;
        if (fixed + 2 * stage > budget) continue;
        p.stages = static_cast<int>((budget - fixed) / stage);
        if (p.stages > kMaxStages) p.stages = kMaxStages;
        smem = fixed + static_cast<size_t>(p.stages) * stage;
        return true;
    }
    return false;
}

}  // namespace

bool fused1x1_supported(const dbp_ctx *ctx, const ConvShape &s, int io) {
    Fused1P p{};
    int rows, nch;
    size_t smem;
    return io == DBP_BF16 && plan_fused1x1(s, ctx->sm_count, p, rows, nch, smem);
}

// dW has been cleared. bf16 dX.
int launch_fused1x1(dbp_ctx *ctx, const void *delta, const void *X, const void *W, const ConvShape &s, unsigned long long seed,
                    const StepSource &step, float *dW, void *dX, int *err_flag) {
    Fused1P p{};
    int rows, nch;
    size_t smem;
    if (!plan_fused1x1(s, ctx->sm_count, p, rows, nch, smem)) return DBP_EUNSUPPORTED;
    p.delta = static_cast<const __nv_bfloat16 *>(delta);
    p.seed = seed;
    p.st = ctx->state;
    p.err_flag = err_flag;
    CUtensorMap map_d, map_w, map_x, map_dx, map_dw;
    const unsigned long long Cin = s.Cin, Cout = s.Cout, HW = p.HW, B = s.B;
    {
        const unsigned long long dims[3] = {HW, Cout, B}, str[2] = {HW * 2, HW * 2 * Cout};
        const unsigned box[3] = {64, static_cast<unsigned>(rows), 1};
        if (!encode_map_bf16(&map_d, delta, 3, dims, str, box)) return fail_cuda("tensor map of delta");
    }
    {
        const unsigned long long dims[2] = {Cin, Cout}, str[1] = {Cin * 2};
        const unsigned box[2] = {64, 64};
        if (!encode_map_bf16(&map_w, W, 2, dims, str, box)) return fail_cuda("tensor map of the weights");
    }
    {
        const unsigned long long dims[3] = {HW, Cin, B}, str[2] = {HW * 2, HW * 2 * Cin};
        const unsigned box_x[3] = {64, static_cast<unsigned>(p.NT), 1}, box_dx[3] = {64, 32, 1};
        if (!encode_map_bf16(&map_x, X, 3, dims, str, box_x)) return fail_cuda("tensor map of the activations");
        if (!encode_map_bf16(&map_dx, dX, 3, dims, str, box_dx)) return fail_cuda("tensor map of dX");
    }
    {
        const unsigned long long dims[2] = {Cin, Cout}, str[1] = {Cin * 4};
        const unsigned box[2] = {32, 32};
        if (!encode_map_f32_sw128(&map_dw, dW, 2, dims, str, box)) return fail_cuda("tensor map of dW");
    }
    auto go = [&](auto kern) -> int {
        if (allow_shared(kern) != cudaSuccess)
            return fail_cuda("shared memory size");
        // One CTA per SM, or as many whole rounds of them as keep a CTA's dW accumulators to kMaxMmas (a chunk is four MMAs)
        const long long most = kMaxMmas / (4 * nch), rounds = (p.ntiles + most * ctx->sm_count - 1) / (most * ctx->sm_count);
        const long long grid = p.ntiles < ctx->sm_count * rounds ? p.ntiles : ctx->sm_count * rounds;
        const long long back = grid * nch;                           // chunks from a CTA's tile to its next one
        p.step_c = static_cast<int>(back % p.cpi);
        auto pairs_z = [](long long elements) { return static_cast<unsigned long long>(elements / 2) * kGamma; };
        const long long image = s.Cout * p.HW;
        p.stage_z = pairs_z(static_cast<long long>(rows) * p.HW);
        p.row64_z = pairs_z(64ll * p.HW);
        p.tile_z = pairs_z(back / p.cpi * image + 64ll * p.step_c) + p.nco * p.stage_z;
        p.wrap_z = pairs_z(64ll * p.cpi) - pairs_z(image);
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(grid)), dim3(kThreadsF), smem, ctx->stream, map_d, map_w, map_x, map_dx,
                                      map_dw, step, p));
    };
    if (rows == 64) return nch == 2 ? go(fused1x1_kernel<64, 2>) : go(fused1x1_kernel<64, 1>);
    return nch == 2 ? go(fused1x1_kernel<128, 2>) : go(fused1x1_kernel<128, 1>);
}

}  // namespace dbp
