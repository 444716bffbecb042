// Backward pass of a small fp32 linear layer in two chained launches (Algorithm 1 with Eqs. (nsd), (qda),
// (qdw)) instead of five: step size + quantization, then both products.
//
// For gradients of a few tens of thousands of elements every separate kernel (statistics, quantizer,
// weight re-layout, dX, dW) is a handful of microseconds of work behind a launch and a dependent wait,
// and the layer is bound by those round trips.
//   1. small_linear_quantize_kernel: ONE cluster of up to eight CTAs holds the whole gradient in registers. The dithers
//      are drawn before the kernel waits for what came before it; every CTA adds up its share, the eight pairs of sums
//      are exchanged through distributed shared memory and added in rank order, so all CTAs hold the same Delta, and
//      each quantizes its share into bf16 codes [B][N rounded up to 8] and counts the non-zero and clipped ones. The
//      first CTA publishes Delta; the second kernel adds up the counts. (Before: every CTA of 4096 elements read the
//      whole gradient for its sums.)
//   2. small_linear_products_kernel: every CTA owns one 64 x 64 tile of dW or of dX and accumulates it
//      on the tensor cores: the codes are exact in bf16, the fp32 operand (X or W) is split into two
//      bf16 pieces (the value rounded to bf16 and what that left over, rounded again: the pair is within
//      2^-17 of the value), so a k-step is two warp-level MMAs with fp32 accumulation; Delta is applied
//      once at the end. Warp-level MMAs (not the CTA-wide ones with accumulators in tensor memory)
//      because a whole tile is a few hundred of them and nothing here can hide a tensor-memory
//      allocation, a commit and a read-back. The dW tiles of column 0 add up the bias gradient.
//      X and W are inputs of the call: a tile's operand of up to 512 reduction indices is loaded, split and laid in shared
//      memory while the first kernel runs; what is left after it is one round trip for the codes and the MMAs.
// The second kernel is launched with programmatic stream serialization: it becomes resident while the first runs.
#include "nsd_common.cuh"
#include "tc_common.cuh"

namespace dbp {

namespace {

using namespace nsd;

constexpr int kThreads = 512;
constexpr int kRows = 64, kCols = 64, kRed = 64;      // output tile and reduction chunk
constexpr int kPitch = 72;                            // halfwords per shared-memory row: a 16-byte multiple whose eight
                                                      // consecutive rows fall into different 16-byte bank groups
constexpr int kChunkTile = 64 * kPitch;               // halfwords of one operand's chunk
constexpr int kMaxChunks = 8;                         // chunks whose operands lie in shared memory at once (three tiles each)
constexpr int kMaxCluster = 8;
constexpr int kMaxVec = 8;                            // 16-byte vectors per thread of the first kernel

__device__ __forceinline__ unsigned smem_addr(const void *p) { return static_cast<unsigned>(__cvta_generic_to_shared(p)); }
// four 8x8 matrices of 16-bit elements from shared memory: lane l gives the address of row l % 8 of matrix l / 8;
// register m of lane (g, tig) receives elements (g, 2 tig) and (g, 2 tig + 1) of matrix m, or, transposed,
// elements (2 tig, g) and (2 tig + 1, g)
__device__ __forceinline__ void ldmatrix_x4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
// D += A (16 x 16, row-major fragments) * B (16 x 8, column-major fragments), bf16 in, fp32 accumulate
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
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

// NV: vectors of four elements per thread (vector i of a thread: blockIdx.x * kThreads + tid + i * all threads)
template <int NV>
__global__ void __launch_bounds__(kThreads)
small_linear_quantize_kernel(const SmallLinP p) {
    __shared__ double red_s[2][kThreads / 32];
    __shared__ double all_s[kMaxCluster][2];
    __shared__ unsigned long long bar_s;           // counts the bytes of the sums that arrive from the cluster's CTAs
    __shared__ float delta_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nctas = gridDim.x;
    const int n = static_cast<int>(p.B * p.N), nvec = (n + 3) / 4, step = nctas * kThreads;
    const int v0 = blockIdx.x * kThreads + tid;
    unsigned long long u[NV][2];
#pragma unroll
    for (int i = 0; i < NV; ++i) dithers_of<4, true>(4ll * (v0 + i * step), p.seed, u[i]);
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
            if (lane < nctas) {                                        // the grid is one cluster: rank = blockIdx.x
                store_remote(&all_s[blockIdx.x][0], &bar_s, lane, a);
                store_remote(&all_s[blockIdx.x][1], &bar_s, lane, b);
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
    for (int i = 0; i < NV; ++i) {
        const int e = 4 * (v0 + i * step);
        if (v0 + i * step < nvec) {
            float f[4];
            unsigned h[2];
            decide<4>(x[i], u[i], inv, f, sat);                        // elements past the end were read as 0: code 0
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
__global__ void __launch_bounds__(kThreads)
small_linear_products_kernel(const SmallLinP p) {
    // per chunk of 64 reduction indices: codes (dX tiles [row][reduction index], dW tiles [reduction index][row], the order
    // they are stored in either way), then rows of X (dW) or W (dX), [reduction index][column], as two bf16 pieces
    extern __shared__ __align__(16) unsigned short tiles_s[];
    __shared__ float db_s[kRows];
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
    if (tid < kRows) db_s[tid] = 0.f;

    // Loads of a chunk: eight consecutive codes per thread, one 16-byte load (dX: row hi, reduction indices
    // lo..lo+7; dW: reduction index hi, rows lo..lo+7), and eight consecutive columns of row hi of X or W.
    const int hi = tid >> 3, lo = (tid & 7) * 8;
    // warp tiling of the 64 x 64 tile: 16 rows x 16 columns per warp (two 16 x 8 accumulators)
    const int wr = (warp >> 2) * 16, wc = (warp & 3) * 16;
    const int g = lane >> 2, tig = lane & 3;
    float acc[2][4] = {}, sum[2][4] = {};
    float dbacc[8] = {};

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
    // Codes outside the tensor read as zero; the padding of a row is cleared when a vector is used (clear_pad), so that the
    // loads of all chunks are in flight together.
    auto load_a = [&](long long r0) {
        const long long bb = is_dw ? r0 + hi : row0 + hi;            // image (row of delta_z)
        const long long jj = is_dw ? row0 + lo : r0 + lo;            // first of eight output channels
        return bb < p.B && jj < p.N ? __ldcg(reinterpret_cast<const uint4 *>(p.codes + bb * p.Np + jj)) : make_uint4(0u, 0u, 0u, 0u);
    };
    auto clear_pad = [&](long long r0, uint4 &v) {
        const long long left = p.N - (is_dw ? row0 + lo : r0 + lo);  // valid codes from the vector's first on
        if (left < 8) {
            unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (2 * i >= left) w[i] = 0u;
                else if (2 * i + 1 >= left) w[i] &= 0xffffu;
            }
            v = make_uint4(w[0], w[1], w[2], w[3]);
        }
    };
    // the addresses this lane hands to the 8x8-matrix loads (lane l: row l % 8 of matrix l / 8)
    const int lm = lane >> 3, lr = lane & 7;
    // A, four matrices: (rows 0-7, k 0-7), (rows 8-15, k 0-7), (rows 0-7, k 8-15), (rows 8-15, k 8-15);
    // dW tiles hold them [k][row] and load them transposed
    const unsigned a_base = smem_addr(tiles_s) + 2u * (is_dw ? static_cast<unsigned>(((lm >> 1) * 8 + lr) * kPitch + wr + (lm & 1) * 8)
                                                             : static_cast<unsigned>((wr + (lm & 1) * 8 + lr) * kPitch + (lm >> 1) * 8));
    const unsigned a_kstep = 2u * (is_dw ? 16u * kPitch : 16u);
    // B, four matrices: (k 0-7, n 0-7), (k 8-15, n 0-7), (k 0-7, n 8-15), (k 8-15, n 8-15), stored [k][n]: transposed loads
    const unsigned b_base = smem_addr(tiles_s) + 2u * static_cast<unsigned>(kChunkTile + ((lm & 1) * 8 + lr) * kPitch + wc + (lm >> 1) * 8);

    // fp32 operand of `count` chunks from r0 on -> its two pieces in shared memory, four chunks' loads in flight
    auto fill_b = [&](long long r0, int count) {
        for (int c0 = 0; c0 < count; c0 += 4) {
            float4 b_reg[4][2];
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c0 + c < count) load_b(r0 + (c0 + c) * kRed, b_reg[c]);
#pragma unroll
            for (int c = 0; c < 4; ++c)
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
                    unsigned short *dst = tiles_s + (c0 + c) * 3 * kChunkTile + kChunkTile + hi * kPitch + lo;
                    *reinterpret_cast<uint4 *>(dst) = make_uint4(h2[0], h2[1], h2[2], h2[3]);
                    *reinterpret_cast<uint4 *>(dst + kChunkTile) = make_uint4(l2[0], l2[1], l2[2], l2[3]);
                }
        }
    };
    // codes of `count` chunks: one round trip for all of them
    auto fill_a = [&](long long r0, int count) {
        {
            uint4 a_reg[kMaxChunks];
#pragma unroll
            for (int c = 0; c < kMaxChunks; ++c)
                a_reg[c] = c < count ? load_a(r0 + c * kRed) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
            for (int c = 0; c < kMaxChunks; ++c)
                if (c < count) {
                    clear_pad(r0 + c * kRed, a_reg[c]);
                    *reinterpret_cast<uint4 *>(tiles_s + c * 3 * kChunkTile + hi * kPitch + lo) = a_reg[c];
                    if (do_db) {
                        const unsigned w[4] = {a_reg[c].x, a_reg[c].y, a_reg[c].z, a_reg[c].w};
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            dbacc[2 * i] += __uint_as_float(w[i] << 16);
                            dbacc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
                        }
                    }
                }
        }
    };
    const int nchunks = static_cast<int>((nred + kRed - 1) / kRed);
    // X and W are inputs of the call: the first chunks' operand is laid out before the first kernel is done
    int count = nchunks < p.chunks ? nchunks : p.chunks;
    fill_b(0, count);
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
    for (int c0 = 0; c0 < nchunks; c0 += p.chunks) {
        count = nchunks - c0 < p.chunks ? nchunks - c0 : p.chunks;
        if (c0 > 0) {
            // an accumulator is truncated when an MMA adds to it: after the 64 MMAs of eight chunks it is added to a sum that rounds
#pragma unroll
            for (int i = 0; i < 8; ++i) { sum[i >> 2][i & 3] += acc[i >> 2][i & 3]; acc[i >> 2][i & 3] = 0.f; }
            __syncthreads();                             // the previous chunks have been used
            fill_b(static_cast<long long>(c0) * kRed, count);
        }
        fill_a(static_cast<long long>(c0) * kRed, count);
        __syncthreads();
        for (int c = 0; c < count; ++c) {
            const unsigned off = 2u * static_cast<unsigned>(c * 3 * kChunkTile);
#pragma unroll
            for (int ks = 0; ks < kRed / 16; ++ks) {
                unsigned a[4], bh[4], bl[4];
                if (is_dw) ldmatrix_x4_trans(a, a_base + off + ks * a_kstep);
                else ldmatrix_x4(a, a_base + off + ks * a_kstep);
                ldmatrix_x4_trans(bh, b_base + off + ks * 2u * 16u * kPitch);
                ldmatrix_x4_trans(bl, b_base + off + 2u * kChunkTile + ks * 2u * 16u * kPitch);
                mma_bf16_16816(acc[0], a, bh[0], bh[1]);
                mma_bf16_16816(acc[1], a, bh[2], bh[3]);
                mma_bf16_16816(acc[0], a, bl[0], bl[1]);
                mma_bf16_16816(acc[1], a, bl[2], bl[3]);
            }
        }
    }

    // the tile, scaled by Delta once: accumulator t holds rows g and g + 8, columns 2 tig, 2 tig + 1 of n-tile t
    float *out = is_dw ? p.dW : p.dX;
#pragma unroll
    for (int tn = 0; tn < 2; ++tn) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long row = row0 + wr + g + 8 * h;
            const long long col = k0 + wc + 8 * tn + 2 * tig;
            if (row >= nrows || col >= p.K) continue;
            float *dst = out + row * p.K + col;
            const float v0 = (sum[tn][2 * h] + acc[tn][2 * h]) * dscale, v1 = (sum[tn][2 * h + 1] + acc[tn][2 * h + 1]) * dscale;
            if ((p.K & 1) == 0) {
                *reinterpret_cast<float2 *>(dst) = make_float2(v0, v1);
            } else {
                dst[0] = v0;
                if (col + 1 < p.K) dst[1] = v1;
            }
        }
    }
    if (do_db) {                                         // threads that share lo hold the same eight rows
#pragma unroll
        for (int i = 0; i < 8; ++i) atomicAdd(&db_s[lo + i], dbacc[i]);     // small integers: exact in any order
        __syncthreads();
        if (tid < kRows && row0 + tid < p.N) p.db[row0 + tid] = db_s[tid] * dscale;
    }
}

}  // namespace

// Shapes the two-launch path takes: a gradient that one cluster holds in registers, and one tile per SM at most. The legacy
// warp-level MMA runs at about 550 multiply-adds per clock and SM here (a 64 x 64 x 16 step with two pieces takes 240
// clocks), so a second tile per SM costs more than the third launch of the CTA-wide kernels (linear_tc.cu). Measured, us,
// this path against that one: 784 -> 300, B 128 (91 tiles): 9.5 against 14.9; 512 -> 1000, B 128 (144): 22.4 against
// 22.8; 1024 -> 100, B 1024 (288): 24.2 against 15.0.
bool small_linear_fits(const dbp_ctx *ctx, long long B, long long N, long long K, bool want_dw, bool want_dx) {
    const long long n = B * N;
    if (n <= 0 || n > 4ll * kMaxCluster * kThreads * kMaxVec || K <= 0 || K > (1ll << 24)) return false;
    const long long tiles_k = (K + kCols - 1) / kCols;
    const long long n_dw = want_dw ? ((N + kRows - 1) / kRows) * tiles_k : 0;
    const long long n_dx = want_dx ? ((B + kRows - 1) / kRows) * tiles_k : 0;
    const long long ctas = n_dw + n_dx;
    return ctas > 0 && ctas <= ctx->sm_count;
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
    p.n_qctas = ctas;
    p.inv_numel = 1.0 / static_cast<double>(n);
    auto kern = per <= 1 ? small_linear_quantize_kernel<1> : per <= 2 ? small_linear_quantize_kernel<2>
              : per <= 5 ? small_linear_quantize_kernel<5> : small_linear_quantize_kernel<kMaxVec>;
    if (int rc = cuda_ok(launch_chained_cluster(kern, static_cast<unsigned>(ctas), static_cast<unsigned>(ctas), dim3(kThreads), 0, ctx->stream, p))) return rc;
    const long long red = (dW && (!dX || B > N)) ? B : N;               // the longest reduction of the tiles
    const long long chunks = (red + kRed - 1) / kRed;
    p.chunks = chunks < kMaxChunks ? static_cast<int>(chunks) : kMaxChunks;
    const size_t smem = static_cast<size_t>(p.chunks) * 3 * kChunkTile * 2;
    if (cudaFuncSetAttribute(small_linear_products_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kMaxChunks * 3 * kChunkTile * 2) != cudaSuccess)
        return fail_cuda("shared memory size");
    return cuda_ok(launch_chained(small_linear_products_kernel, dim3(static_cast<unsigned>(p.n_dw + p.n_dx)), dim3(kThreads), smem,
                                  ctx->stream, p));
}

}  // namespace dbp
