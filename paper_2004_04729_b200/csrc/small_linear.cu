// Backward pass of a small fp32 linear layer in two chained launches (Algorithm 1 with Eqs. (nsd), (qda),
// (qdw)) instead of five: step size + quantization, then both products.
//
// For gradients of a few tens of thousands of elements every separate kernel (statistics, quantizer,
// weight re-layout, dX, dW) is a handful of microseconds of work behind a launch and a dependent wait,
// and the layer is bound by those round trips.
//   1. small_linear_quantize_kernel: one to five clusters of up to eight CTAs. Every cluster holds the whole gradient in
//      registers. The dithers are drawn before the kernel waits for what came before it; every CTA adds up its share, the
//      cluster's pairs of sums are exchanged through distributed shared memory and added in rank order, so all CTAs hold the
//      same Delta, and each cluster quantizes its part of the vectors into bf16 codes [B][N rounded up to 8] and counts the non-zero and
//      clipped ones. The first CTA publishes Delta; the second kernel adds up the counts.
//   2. small_linear_products_kernel: every CTA owns one 64 x 64 tile of dW or of dX and accumulates it on the tensor cores:
//      the codes are exact in bf16, the fp32 operand (X or W) is split into two bf16 pieces (the value rounded to bf16 and
//      what that left over, rounded again: the pair is within 2^-17 of the value), whose panels lie beside one another as one
//      operand of 128 columns; Delta is applied once at the end. The dW tiles of column 0 add up the bias gradient.
//      X and W are inputs of the call: a tile's operand of up to 512 reduction indices is loaded, split and laid in shared
//      memory while the first kernel runs; what is left after it is one tiled copy per chunk of codes and the MMAs.
// The second kernel is launched with programmatic stream serialization: it becomes resident while the first runs.
//
// Bound by the chain: two kernel boundaries and, for 784 -> 300 at batch 128 in thousands of clocks, loads and sums 2.4, Delta 1.2,
// decisions 0.9 (one cluster: 2.0), codes by the copy engine and their MMAs, then the tile through shared memory to whole
// lines. With codes loaded and laid out by the threads (3.7), warp-level MMAs (4.5 of a five-chunk tile) and stores of 32 rows an
// instruction (1.5) the call took 9.45 us; it takes 7.95. 784-300-100-10, batch 256: 26.6, 22.6. Registers held to 80 or 64, so that the
// first kernel of the next call fits beside the second: 8.03, 8.73.
#include "nsd_common.cuh"
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace nsd;

constexpr int kThreads = 512;
constexpr int kRows = 64, kCols = 64, kRed = 64;      // output tile and reduction chunk
constexpr int kChunkTile = 64 * 128;                  // bytes of one operand's chunk: 64 rows of 64 bf16, 16-byte pieces swizzled by the row
constexpr int kMaxChunks = 8;                         // chunks whose operands lie in shared memory at once (three tiles each)
constexpr int kTmemCols = 128;                        // accumulators: 64 columns of the high pieces' products, 64 of the low ones'
constexpr int kMaxCluster = 8;
constexpr int kMaxVec = 8;                            // 16-byte vectors per thread of the first kernel

__device__ __forceinline__ unsigned smem_addr(const void *p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
// sixteen accumulator columns (the caller waits)
__device__ __forceinline__ void tmem_ld16(unsigned taddr, unsigned (&r)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                   "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]) : "r"(taddr));
}

struct SmallLinP {
    const float *delta, *X, *W;   // [B][N], [B][K], [N][K]
    const uint8_t *mask;          // not null: delta is delta_a and the gradient is delta_a where mask != 0, else 0
    const float *delta_in;        // used when scale <= 0
    float scale;
    long long B, N, K, Np;        // Np: N rounded up to 8, the row pitch of the codes
    unsigned long long seed;
    float *dW, *dX, *db;          // any may be null (not both products)
    DeviceState *st;
    float *delta_set;             // second place the step size goes to (may be null)
    unsigned short *codes;        // bf16 [B][Np]
    unsigned *slots;              // one non-zero count per warp of the first kernel
    double inv_numel;
    int tiles_k, n_dw, n_dx, n_qctas;
    int vec4;                     // K % 4 == 0: 16-byte accesses along K
    int chunks;                   // chunks of the reduction in shared memory at once
};

// ---------------------------------------------------------------- step size and codes
// stores a double at the same place of another CTA's shared memory; its 8 bytes are counted on that CTA's barrier
__device__ __forceinline__ void store_remote(double *p, unsigned long long *bar, unsigned rank, double v) {
    unsigned addr, baddr;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_addr(p)), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(baddr) : "r"(smem_addr(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];"
                 ::"r"(addr), "l"(__double_as_longlong(v)), "r"(baddr) : "memory");
}

// NV: vectors of four elements per thread of a cluster (vector i of a thread: rank * kThreads + tid + i * all threads). There are
// NCL clusters; every one of them has the whole gradient for the sums, and decides the vectors i = its number, + NCL, ...
// (see the head of this file)
template <int NV, int NCL>
__global__ void __launch_bounds__(kThreads)
small_linear_quantize_kernel(const SmallLinP p) {
    constexpr int ND = (NV + NCL - 1) / NCL;       // vectors a thread decides, at most
    __shared__ double red_s[2][kThreads / 32];
    __shared__ double all_s[kMaxCluster][2];
    __shared__ unsigned long long bar_s;           // counts the bytes of the sums that arrive from the cluster's CTAs
    __shared__ float delta_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nctas = gridDim.x / NCL;
    const int cluster = NCL == 1 ? 0 : static_cast<int>(blockIdx.x) / nctas, rank = static_cast<int>(blockIdx.x) - cluster * nctas;
    const int n = static_cast<int>(p.B * p.N), nvec = (n + 3) / 4, step = nctas * kThreads;
    const int v0 = rank * kThreads + tid;
    unsigned long long u[ND][2];
#pragma unroll
    for (int d = 0; d < ND; ++d) dithers_of<4, true>(4ll * (v0 + (cluster + d * NCL) * step), p.seed, u[d]);
    if (tid == 0) {
        tc::mbar_init(&bar_s, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc::mbar_expect_tx(&bar_s, 16u * nctas);
    }
    // every CTA's barrier is there before anybody's sums leave (long before: this is in front of the wait)
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    chain_wait();
    chain_release();

    float x[NV][4];
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        const int e = 4 * (v0 + i * step);
        if (e + 4 <= n) {
            const float4 q = __ldcg(reinterpret_cast<const float4 *>(p.delta + e));
            x[i][0] = q.x; x[i][1] = q.y; x[i][2] = q.z; x[i][3] = q.w;
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) x[i][j] = e + j < n ? __ldcg(p.delta + e + j) : 0.f;
        }
    }
    if (p.mask != nullptr) {
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = 4 * (v0 + i * step);
            if (e + 4 <= n) {
                const uchar4 m = __ldg(reinterpret_cast<const uchar4 *>(p.mask + e));
                x[i][0] = m.x ? x[i][0] : 0.f; x[i][1] = m.y ? x[i][1] : 0.f; x[i][2] = m.z ? x[i][2] : 0.f; x[i][3] = m.w ? x[i][3] : 0.f;
            } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (e + j < n && !__ldg(p.mask + e + j)) x[i][j] = 0.f;
            }
        }
    }
    // step size: shifted moments about the first element, fp32 inside a vector, fp64 across
    float delta;
    bool nonfinite = false;
    if (p.scale > 0.f) {
        const float pivot = (p.mask == nullptr || __ldg(p.mask)) ? __ldcg(p.delta) : 0.f;
        double d1 = 0.0, d2 = 0.0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int e = 4 * (v0 + i * step);
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float c = e + j < n ? x[i][j] - pivot : 0.f;
                s1 += c;
                s2 = fmaf(c, c, s2);
            }
            d1 += static_cast<double>(s1);
            d2 += static_cast<double>(s2);
        }
        d1 = warp_sum(d1);
        d2 = warp_sum(d2);
        if (lane == 0) { red_s[0][warp] = d1; red_s[1][warp] = d2; }
        __syncthreads();
        if (warp == 0) {
            // sixteen partial sums of each moment in the two halves of the warp
            double v = red_s[lane >> 4][lane & 15];
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
            const double a = __shfl_sync(kFull, v, 0), b = __shfl_sync(kFull, v, 16);
            if (lane < nctas) {
                store_remote(&all_s[rank][0], &bar_s, lane, a);
                store_remote(&all_s[rank][1], &bar_s, lane, b);
            }
        }
        // (a CTA ends only after all sums have arrived here, so nothing is still on its way to it then)
        const bool here = tc::mbar_wait(&bar_s, 0, &p.st->tc_timeout);
        if (tid == 0) {
            double a = 0.0, b = 0.0;
#pragma unroll
            for (int r = 0; r < kMaxCluster; ++r)
                if (r < nctas) { a += all_s[r][0]; b += all_s[r][1]; }
            if (!here) a = b = 0.0;
            delta = 0.f;
            if (!isfinite(a) || !isfinite(b)) {
                nonfinite = true;
            } else {
                const double mean = a * p.inv_numel;
                double var = b * p.inv_numel - mean * mean;
                if (var < 0.0) var = 0.0;
                delta = static_cast<float>(static_cast<double>(p.scale) * sqrt(var));
            }
            delta_s = delta;
        }
        __syncthreads();
        delta = delta_s;
    } else {
        delta = __ldcg(p.delta_in);
    }
    const bool live = (delta > 0.f) && (delta < __int_as_float(0x7f800000));
    const float inv = live ? __fdiv_rn(1.0f, delta) : 0.f;             // Delta = 0: every code 0

    unsigned nz2 = 0, sat = 0;
    const unsigned N = static_cast<unsigned>(p.N);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        const int i = cluster + d * NCL, e = 4 * (v0 + i * step);
        if (i < NV && v0 + i * step < nvec) {
            float f[4], xi[4];
            unsigned h[2];
#pragma unroll
            for (int k = 0; k < NCL; ++k)                              // (an index that is no constant would put x into memory)
                if (d * NCL + k < NV && k == cluster)
#pragma unroll
                    for (int j = 0; j < 4; ++j) xi[j] = x[d * NCL + k < NV ? d * NCL + k : 0][j];
            decide<4>(xi, u[d], inv, f, sat);                          // elements past the end were read as 0: code 0
            pack_bf16<4>(f, h);
            count_pairs<4>(h, nz2);
            const unsigned b = static_cast<unsigned>(e) / N, j = static_cast<unsigned>(e) - b * N;
            unsigned short *dst = p.codes + b * p.Np + j;
            if ((N & 3u) == 0) {                                       // four codes of one row
                *reinterpret_cast<uint2 *>(dst) = make_uint2(h[0], h[1]);
            } else {
                unsigned jj = j;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (e + k < n) *dst = static_cast<unsigned short>(h[k >> 1] >> (16 * (k & 1)));
                    ++dst;
                    if (++jj == N) { jj = 0; dst += p.Np - N; }
                }
            }
        }
    }
    const unsigned nnz = __reduce_add_sync(kFull, pairs_total(nz2));
    sat = __reduce_add_sync(kFull, live ? sat : 0u);
    // The counts of the warps are added up by the products kernel, which runs when all of them are done. Every CTA holds
    // the same Delta, so the first one publishes it.
    if (lane == 0) {
        p.slots[blockIdx.x * (kThreads / 32) + warp] = nnz;
        if (sat) atomicAdd(&p.st->saturated, static_cast<unsigned long long>(sat));
    }
    if (blockIdx.x == 0 && tid == 0) {
        p.st->delta = delta;
        if (nonfinite) p.st->nonfinite = 1;
        if (p.delta_set) *p.delta_set = delta;
    }
}

// ---------------------------------------------------------------- both products
__global__ void __launch_bounds__(kThreads, 1)
small_linear_products_kernel(const __grid_constant__ CUtensorMap map_q, const SmallLinP p) {
    // per chunk of 64 reduction indices: codes (dX tiles [row][reduction index], dW tiles [reduction index][row], the order
    // they are stored in either way), then rows of X (dW) or W (dX), [reduction index][column], as two bf16 pieces
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *const tiles_s = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ unsigned long long codes_in[kMaxChunks], mma_done;
    __shared__ unsigned tmem_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    const int t = blockIdx.x;
    const bool is_dw = t < p.n_dw;
    const int tt = is_dw ? t : t - p.n_dw;
    const int rt = tt / p.tiles_k, kt = tt - rt * p.tiles_k;
    const long long row0 = static_cast<long long>(rt) * kRows;      // first output row: j (dW) or b (dX)
    const long long k0 = static_cast<long long>(kt) * kCols;
    const long long nrows = is_dw ? p.N : p.B;                       // output rows in all
    const long long nred = is_dw ? p.B : p.N;                        // reduction length
    const float *Bsrc = is_dw ? p.X : p.W;                           // [nred][K]
    const bool do_db = is_dw && kt == 0 && p.db != nullptr;
    if (tid == 0) {
        for (int c = 0; c < kMaxChunks; ++c) tc::mbar_init(&codes_in[c], 1);
        tc::mbar_init(&mma_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        tc::tma_prefetch_desc(&map_q);
    }
    if (warp == 1) tc::tmem_alloc(&tmem_s, kTmemCols);

    // Of a chunk a thread loads eight consecutive columns of row hi of X or W.
    const int hi = tid >> 3, lo = (tid & 7) * 8;
    const int place = hi * 128 + (((tid & 7) ^ (hi & 7)) << 4);      // where they lie in a tile
    // Of the accumulators' lanes the first 64 are rows of the tile: the warps of the first two lane quarters read them, sixteen
    // columns each.
    const int q = warp & 3, c16 = (warp >> 2) * 16;
    float sum[16] = {};

    auto load_b = [&](long long r0, float4 (&b_reg)[2]) {
        const long long r = r0 + hi;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const long long c = k0 + lo + 4 * h;
            if (r < nred) {
                const float *src = Bsrc + r * p.K + c;
                if (p.vec4) {
                    if (c < p.K) v = __ldg(reinterpret_cast<const float4 *>(src));
                } else {
                    if (c + 0 < p.K) v.x = __ldg(src + 0);
                    if (c + 1 < p.K) v.y = __ldg(src + 1);
                    if (c + 2 < p.K) v.z = __ldg(src + 2);
                    if (c + 3 < p.K) v.w = __ldg(src + 3);
                }
            }
            b_reg[h] = v;
        }
    };
    // fp32 operand of `count` chunks from r0 on -> its two pieces in shared memory, two chunks' loads in flight
    auto fill_b = [&](long long r0, int count) {
        for (int c0 = 0; c0 < count; c0 += 2) {
            float4 b_reg[2][2];
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (c0 + c < count) load_b(r0 + (c0 + c) * kRed, b_reg[c]);
#pragma unroll
            for (int c = 0; c < 2; ++c)
                if (c0 + c < count) {
                    const float v[8] = {b_reg[c][0].x, b_reg[c][0].y, b_reg[c][0].z, b_reg[c][0].w,
                                        b_reg[c][1].x, b_reg[c][1].y, b_reg[c][1].z, b_reg[c][1].w};
                    unsigned h2[4], l2[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const __nv_bfloat162 hh = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
                        const float2 hf = __bfloat1622float2(hh);
                        const __nv_bfloat162 ll = __floats2bfloat162_rn(v[2 * i] - hf.x, v[2 * i + 1] - hf.y);
                        h2[i] = *reinterpret_cast<const unsigned *>(&hh);
                        l2[i] = *reinterpret_cast<const unsigned *>(&ll);
                    }
                    unsigned char *dst = tiles_s + (c0 + c) * 3 * kChunkTile + kChunkTile + place;
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(h2[0], h2[1], h2[2], h2[3]);
                    *reinterpret_cast<uint4 *>(dst + kChunkTile) = make_uint4(l2[0], l2[1], l2[2], l2[3]);
                }
        }
    };
    const int nchunks = static_cast<int>((nred + kRed - 1) / kRed);
    // X and W are inputs of the call: the first chunks' operand is laid out before the first kernel is done
    int count = nchunks < p.chunks ? nchunks : p.chunks;
    fill_b(0, count);
    tc::fence_async_proxy();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const unsigned tmem = tmem_s;
    chain_wait();
    chain_release();
    const float delta = __ldcg(&p.st->delta);
    const float dscale = (delta > 0.f && delta < __int_as_float(0x7f800000)) ? delta : 0.f;
    if (blockIdx.x == 0 && warp == 0) {                  // nnz of the step: the first kernel's per-CTA counts
        unsigned long long total = 0;
        for (int i = lane; i < p.n_qctas * (kThreads / 32); i += 32) total += __ldcg(p.slots + i);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(kFull, total, o);
        if (lane == 0) p.st->nnz = total;
    }
    // A chunk's codes come as one tiled copy, rows of 64 swizzled as an MMA reads them; outside the tensor they are zero. They are
    // used as they lie (dX: K-major, 16 reduction indices 32 bytes further; dW: MN-major, 16 rows = 2048 bytes further); X or
    // W MN-major, the low pieces' panel as columns 64-127. An MMA has 128 rows and the tile 64: the upper ones are whatever
    // follows the codes (dX) or the same codes (dW), and nobody reads them.
    const unsigned idesc = tc::make_idesc(128, 128, is_dw, true);
    const unsigned long long a_desc = tc::make_desc(smem_addr(tiles_s), is_dw ? 0 : 16, 1024);
    const unsigned long long b_desc = tc::make_desc(smem_addr(tiles_s) + kChunkTile, kChunkTile, 1024);
    const unsigned a_step = is_dw ? 128 : 2;
    const int j0 = static_cast<int>(row0), jr = static_cast<int>(kRed);
    float dbacc[8] = {};
    unsigned parity = 0;
    bool ok = true;
    for (int c0 = 0; c0 < nchunks && ok; c0 += p.chunks) {
        count = nchunks - c0 < p.chunks ? nchunks - c0 : p.chunks;
        if (c0 > 0) {
            fill_b(static_cast<long long>(c0) * kRed, count);
            tc::fence_async_proxy();
            tc::tc_fence_before();
            __syncthreads();
            tc::tc_fence_after();
        }
        if (warp == 0) {
            if (tc::elect_one())
                for (int c = 0; c < count; ++c) {
                    tc::mbar_expect_tx(&codes_in[c], kChunkTile);
                    tc::tma_load_2d(tiles_s + c * 3 * kChunkTile, &map_q, is_dw ? j0 : (c0 + c) * jr, is_dw ? (c0 + c) * jr : j0, &codes_in[c]);
                }
            __syncwarp();
        } else if (warp == 1) {
            for (int c = 0; c < count && ok; ++c) {
                ok = __all_sync(kFull, tc::mbar_wait(&codes_in[c], parity, &p.st->tc_timeout));
                tc::tc_fence_after();
                const unsigned long long ad = a_desc + static_cast<unsigned>(c * 3 * (kChunkTile >> 4)), bd = b_desc + static_cast<unsigned>(c * 3 * (kChunkTile >> 4));
                if (ok && tc::elect_one())
#pragma unroll
                    for (int k = 0; k < kRed / 16; ++k) tc::mma_bf16(tmem, ad + k * a_step, bd + 128 * k, idesc, c + k ? 1u : 0u);
            }
            if (ok && tc::elect_one()) tc::mma_commit(&mma_done);
            __syncwarp();
        }
        if (do_db)                                       // beside the MMAs
            for (int c = 0; c < count && ok; ++c) {
                ok = tc::mbar_wait(&codes_in[c], parity, &p.st->tc_timeout);       // (the copy's bytes are seen by who waits for it)
                const uint4 v = *reinterpret_cast<const uint4 *>(tiles_s + c * 3 * kChunkTile + place);
                const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    dbacc[2 * i] += __uint_as_float(w[i] << 16);
                    dbacc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
                }
            }
        // an accumulator is truncated when an MMA adds to it: after the MMAs of eight chunks it is added to a sum that rounds
        // (and the chunks' places are written again only when they have been read)
        ok = tc::mbar_wait(&mma_done, parity, &p.st->tc_timeout) && ok;
        tc::tc_fence_after();
        parity ^= 1u;
        __syncwarp();
        if (q < 2) {
            unsigned h[16], l[16];
            const unsigned at = tmem + (static_cast<unsigned>(q * 32) << 16) + c16;
            tmem_ld16(at, h);
            tmem_ld16(at + 64, l);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int i = 0; i < 16; ++i) sum[i] += __uint_as_float(h[i]) + __uint_as_float(l[i]);
            tc::tc_fence_before();
        }
        ok = __syncthreads_and(ok) != 0;
    }
    if (warp == 1) tc::tmem_dealloc(tmem, kTmemCols);

    // The tile, scaled by Delta once: a thread has sixteen columns of a row. Through shared memory (16-byte pieces swizzled by the
    // row), so that lanes store along the rows: 32 rows an instruction took 1500 clocks.
    if (ok) {
        float4 *const stg = reinterpret_cast<float4 *>(tiles_s);
        if (q < 2) {
            const int r = q * 32 + lane;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                stg[r * 16 + (((c16 >> 2) + i) ^ (r & 7))] = make_float4(sum[4 * i] * dscale, sum[4 * i + 1] * dscale, sum[4 * i + 2] * dscale, sum[4 * i + 3] * dscale);
        }
        __syncthreads();
        float *const out = is_dw ? p.dW : p.dX;
        if (p.vec4) {
            const long long col = k0 + (lane & 15) * 4;
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const int r = warp * 4 + 2 * i + (lane >> 4);
                if (row0 + r < nrows && col < p.K)
                    *reinterpret_cast<float4 *>(out + (row0 + r) * p.K + col) = stg[r * 16 + ((lane & 15) ^ (r & 7))];
            }
        } else {                                         // rows that start anywhere: element by element along them
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int r = warp * 4 + (i >> 1), c = (i & 1) * 32 + lane;
                if (row0 + r < nrows && k0 + c < p.K)
                    out[(row0 + r) * p.K + k0 + c] = reinterpret_cast<const float *>(stg)[r * 64 + (((c >> 2) ^ (r & 7)) << 2) + (c & 3)];
            }
        }
    }
    if (do_db && ok) {
        // Threads that share lo hold the same eight rows: four of a warp, then the warps in shared memory behind the staged tile (small
        // integers: exact in any order). 64 atomic additions to each of 64 places instead took 4 us: 784 -> 300, batch 128, with
        // its bias gradient 12.3 us, 7.8 so.
        float *const part = reinterpret_cast<float *>(tiles_s) + kRows * kCols;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            float v = dbacc[i] + __shfl_xor_sync(kFull, dbacc[i], 8);
            v += __shfl_xor_sync(kFull, v, 16);
            if (lane < 8) part[warp * kRows + lo + i] = v;
        }
        __syncthreads();
        if (tid < kRows && row0 + tid < p.N) {
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kThreads / 32; ++w) v += part[w * kRows + tid];
            p.db[row0 + tid] = v * dscale;
        }
    }
}

}  // namespace

// Shapes the two-launch path takes: a gradient that one cluster holds in registers, and one tile per SM at most, or two of
// reductions that lie in shared memory at once and are at most ten chunks of 64 an SM, all tiles together. More cost more
// than the third launch of the CTA-wide kernels (linear_tc.cu).
// us, this path against that one, fp32 as (batch, outputs, inputs): (128, 300, 784), 91 tiles: 7.95, 14.9; (128, 1000, 512), 144:
// 17.1, 22.4; (128, 512, 1024), 160: 14.0, 16.4; (300, 300, 1500), 240 of five chunks, 8.1 an SM: 14.7, 15.4; (288, 262, 1812), 290, 9.8:
// 15.6, 16.5; (64, 512, 2048), 288: 13.9, 15.7; more chunks: (256, 512, 1500), 288, 10.4: 17.1, 15.5; (512, 256, 1500), 288, 10.4: 15.6, 14.8;
// (327, 384, 1496), 288, 11.7: 16.8, 15.2;
// two rounds of chunks: (1024, 100, 1024), 288: 16.0, 14.3; (1000, 64, 1000), 272: 14.7, 13.1; three tiles: (500, 128, 2048),
// 320: 15.5, 14.0.
bool small_linear_fits(const dbp_ctx *ctx, long long B, long long N, long long K, bool want_dw, bool want_dx) {
    const long long n = B * N;
    if (n <= 0 || n > 4ll * kMaxCluster * kThreads * kMaxVec || K <= 0 || K > (1ll << 24)) return false;
    const long long tiles_k = (K + kCols - 1) / kCols;
    const long long n_dw = want_dw ? ((N + kRows - 1) / kRows) * tiles_k : 0;
    const long long n_dx = want_dx ? ((B + kRows - 1) / kRows) * tiles_k : 0;
    const long long ctas = n_dw + n_dx;
    const long long red = want_dw && (!want_dx || B > N) ? B : N;
    const long long chunks = n_dw * ((B + kRed - 1) / kRed) + n_dx * ((N + kRed - 1) / kRed);
    return ctas > 0 && (ctas <= ctx->sm_count || (ctas <= 2 * ctx->sm_count && red <= kMaxChunks * kRed && chunks <= 10 * ctx->sm_count));
}

int launch_small_linear(dbp_ctx *ctx, const float *delta, const float *X, const float *W, long long B, long long N,
                        long long K, unsigned long long seed, float scale, const float *delta_in, float *dW, float *dX,
                        float *db, float *delta_set, const uint8_t *mask) {
    SmallLinP p{};
    p.delta = delta; p.X = X; p.W = W; p.delta_in = delta_in; p.scale = scale; p.mask = mask;
    p.B = B; p.N = N; p.K = K; p.Np = (N + 7) / 8 * 8; p.seed = seed;
    p.dW = dW; p.dX = dX; p.db = dW ? db : nullptr;
    p.st = ctx->state; p.delta_set = delta_set;
    const int k = ctx->code_set;
    if (int rc = ws_reserve(ctx, ctx->codes16[k], static_cast<size_t>(B) * p.Np * 2 + 64)) return rc;
    p.codes = static_cast<unsigned short *>(ctx->codes16[k].ptr);
    p.slots = reinterpret_cast<unsigned *>(ctx->partials);
    p.tiles_k = static_cast<int>((K + kCols - 1) / kCols);
    p.n_dw = dW ? static_cast<int>((N + kRows - 1) / kRows) * p.tiles_k : 0;
    p.n_dx = dX ? static_cast<int>((B + kRows - 1) / kRows) * p.tiles_k : 0;
    p.vec4 = (K % 4 == 0) ? 1 : 0;
    // the cluster grows before the vectors per thread do
    const long long n = B * N, nvec = (n + 3) / 4;
    int ctas = 1;
    while (ctas < kMaxCluster && ctas * kThreads < nvec) ctas *= 2;
    const int per = static_cast<int>((nvec + ctas * kThreads - 1) / (ctas * kThreads));
    const int ncl = per <= 1 ? 1 : per <= 2 ? 2 : per <= 5 ? 5 : 4;
    p.n_qctas = ctas * ncl;
    p.inv_numel = 1.0 / static_cast<double>(n);
    auto kern = per <= 1 ? small_linear_quantize_kernel<1, 1> : per <= 2 ? small_linear_quantize_kernel<2, 2>
              : per <= 5 ? small_linear_quantize_kernel<5, 5> : small_linear_quantize_kernel<kMaxVec, 4>;
    if (int rc = cuda_ok(launch_chained_cluster(kern, static_cast<unsigned>(ctas * ncl), static_cast<unsigned>(ctas), dim3(kThreads), 0, ctx->stream, p))) return rc;
    CUtensorMap map_q;
    {
        const unsigned long long dims[2] = {static_cast<unsigned long long>(N), static_cast<unsigned long long>(B)};
        const unsigned long long str[1] = {static_cast<unsigned long long>(p.Np) * 2};
        const unsigned box[2] = {kRed, kRows};
        if (!tc::encode_map_bf16(&map_q, p.codes, 2, dims, str, box)) return fail_cuda("tensor map of the codes");
    }
    const long long red = (dW && (!dX || B > N)) ? B : N;               // the longest reduction of the tiles
    const long long chunks = (red + kRed - 1) / kRed;
    p.chunks = chunks < kMaxChunks ? static_cast<int>(chunks) : kMaxChunks;
    const size_t smem = static_cast<size_t>(p.chunks) * 3 * kChunkTile + 1024;
    if (cudaFuncSetAttribute(small_linear_products_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxChunks * 3 * kChunkTile + 1024) != cudaSuccess)
        return fail_cuda("shared memory size");
    return cuda_ok(launch_chained(small_linear_products_kernel, dim3(static_cast<unsigned>(p.n_dw + p.n_dx)), dim3(kThreads), smem,
                                  ctx->stream, map_q, p));
}

}  // namespace dbp
