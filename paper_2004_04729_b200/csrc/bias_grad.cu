// Bias gradients from the bf16 codes the tensor-core products read: db[c] = Delta * sum of channel c's codes.
//
// The sums are integers and are added as integers (the order does not matter), Delta is applied once. A reduction is
// split over blocks; the last block of a channel adds up the parts and puts its counter back to zero.
//
// `beside`: the kernel before this one on the stream writes nothing this one reads and has let it start when all of its
// CTAs had seen everything before them complete. Such a call works first, beside that kernel (a product, bound by the
// tensor pipe or by its stores), and waits for it only before it ends, so that whatever comes behind waits for both. One block does:
// where all did, the blocks that the product's CTAs leave room for held it until the product was done and the others ran behind it
// (1024 -> 4096 bf16, batch 4096, with its bias gradient: 85.2 us, 79.4 so).
#include "dbp_internal.cuh"

namespace dbp {

namespace {

constexpr long long kMaxGroups = 16384;           // counters in the workspace: reductions over more groups are not split

// db[j] = Delta * sum_b q[b][j] from the bf16 codes [B][pitch]. A block owns 64 columns and a range of rows, a thread
// eight of the columns and every 32nd row, four 16-byte loads in flight. A thread's own sum is exact in fp32 (integers
// below 2^24 up to four million rows of full-scale codes); the threads' and the blocks' sums are added as integers, the
// last block of a column group adding up the ranges and putting its counter back to zero.
__global__ void __launch_bounds__(256)
column_sums_kernel(const unsigned short *__restrict__ codes, long long rows, int cols, long long pitch, long long per_split,
                   int *__restrict__ partials, unsigned *__restrict__ tickets, const float *__restrict__ delta_p,
                   float *__restrict__ db, int beside) {
    __shared__ int sum_s[64];
    __shared__ bool is_last;
    if (threadIdx.x < 64) sum_s[threadIdx.x] = 0;
    __syncthreads();
    if (!beside) chain_wait();
    chain_release();
    const int c0 = blockIdx.x * 64 + (threadIdx.x & 7) * 8;
    const long long r1 = (blockIdx.y + 1) * per_split < rows ? (blockIdx.y + 1) * per_split : rows;
    float facc[8] = {};
    if (c0 < cols) {
        auto add = [&](const uint4 &v) {
            const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                facc[2 * i] += __uint_as_float(w[i] << 16);
                facc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);
            }
        };
        long long r = blockIdx.y * per_split + (threadIdx.x >> 3);
        const unsigned short *src = codes + r * pitch + c0;
        for (; r + 96 < r1; r += 128, src += 128 * pitch) {
            uint4 v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = __ldcg(reinterpret_cast<const uint4 *>(src + 32 * u * pitch));
#pragma unroll
            for (int u = 0; u < 4; ++u) add(v[u]);
        }
        for (; r < r1; r += 32, src += 32 * pitch) add(__ldcg(reinterpret_cast<const uint4 *>(src)));
    }
    // the four row groups of a warp, then the warps (padding columns may hold anything; they are not stored)
    int acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        acc[i] = static_cast<int>(facc[i]);
        acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 8);
        acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
    }
    if ((threadIdx.x & 31) < 8)
#pragma unroll
        for (int i = 0; i < 8; ++i) atomicAdd(&sum_s[(threadIdx.x & 7) * 8 + i], acc[i]);
    __syncthreads();
    const int c = blockIdx.x * 64 + threadIdx.x;
    int total = threadIdx.x < 64 ? sum_s[threadIdx.x] : 0;
    if (gridDim.y > 1) {
        if (threadIdx.x < 64) __stcg(partials + (blockIdx.y * static_cast<long long>(gridDim.x) + blockIdx.x) * 64 + threadIdx.x, total);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) {
            is_last = atomicAdd(tickets + blockIdx.x, 1u) == gridDim.y - 1;
            if (is_last) tickets[blockIdx.x] = 0u;
        }
        __syncthreads();
        if (is_last && threadIdx.x < 64) {
            __threadfence();
            total = 0;
#pragma unroll 4
            for (unsigned s = 0; s < gridDim.y; ++s)
                total += __ldcg(partials + (s * static_cast<long long>(gridDim.x) + blockIdx.x) * 64 + threadIdx.x);
        }
        if (is_last && threadIdx.x < 64 && c < cols) db[c] = static_cast<float>(total) * (*delta_p);
    } else if (threadIdx.x < 64 && c < cols) {
        db[c] = static_cast<float>(total) * (*delta_p);
    }
    if (beside && blockIdx.x == 0 && blockIdx.y == 0) chain_wait();
}

// Planes [image][channel][pitch]: a block owns one channel and a range of images, a warp one plane at a time.
__global__ void __launch_bounds__(256)
plane_sums_kernel(const unsigned short *__restrict__ codes, int B, long long hw, long long pitch, int per_split,
                  int *__restrict__ partials, unsigned *__restrict__ tickets, const float *__restrict__ delta_p,
                  float *__restrict__ db, int beside) {
    __shared__ int sum_s[8];
    if (!beside) chain_wait();
    chain_release();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int b1 = (blockIdx.y + 1) * per_split < B ? (blockIdx.y + 1) * per_split : B;
    int acc = 0;
    for (int b = blockIdx.y * per_split + warp; b < b1; b += 8) {
        const unsigned short *src = codes + (static_cast<long long>(b) * gridDim.x + blockIdx.x) * pitch;
        for (long long p0 = lane * 8; p0 < hw; p0 += 256) {
            const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(src + p0));
            const unsigned w[4] = {v.x, v.y, v.z, v.w};
            float s = 0.f;
#pragma unroll
            for (int i = 0; i < 4; ++i) {                          // the padding of a plane may hold anything
                if (p0 + 2 * i < hw) s += __uint_as_float(w[i] << 16);
                if (p0 + 2 * i + 1 < hw) s += __uint_as_float(w[i] & 0xffff0000u);
            }
            acc += static_cast<int>(s);
        }
    }
    acc = __reduce_add_sync(0xffffffffu, acc);
    if (lane == 0) sum_s[warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        int total = 0;
        for (int w = 0; w < 8; ++w) total += sum_s[w];
        bool last = true;
        if (gridDim.y > 1) {
            __stcg(partials + static_cast<long long>(blockIdx.y) * gridDim.x + blockIdx.x, total);
            __threadfence();
            last = atomicAdd(tickets + blockIdx.x, 1u) == gridDim.y - 1;
            if (last) {
                tickets[blockIdx.x] = 0u;
                __threadfence();
                total = 0;
                for (unsigned s = 0; s < gridDim.y; ++s) total += __ldcg(partials + static_cast<long long>(s) * gridDim.x + blockIdx.x);
            }
        }
        if (last) db[blockIdx.x] = static_cast<float>(total) * (*delta_p);
    }
    if (beside && blockIdx.x == 0 && blockIdx.y == 0) chain_wait();
}

// counters (zero between calls) at the start of the workspace, partial sums after them
int sums_workspace(dbp_ctx *ctx, size_t sums, int **partials, unsigned **tickets, bool *beside) {
    const size_t had = ctx->db_sums.bytes, counter_bytes = kMaxGroups * sizeof(unsigned);
    if (int rc = ws_reserve(ctx, ctx->db_sums, counter_bytes + sums * sizeof(int))) return rc;
    if (ctx->db_sums.bytes != had) {
        if (cudaMemsetAsync(ctx->db_sums.ptr, 0, counter_bytes, ctx->stream) != cudaSuccess)
            return fail_cuda("clearing the counters of the bias gradient");
        *beside = false;                           // the memset lies between this kernel and the one before
    }
    *tickets = static_cast<unsigned *>(ctx->db_sums.ptr);
    *partials = reinterpret_cast<int *>(static_cast<unsigned char *>(ctx->db_sums.ptr) + counter_bytes);
    return DBP_OK;
}

}  // namespace

// codes: bf16 [rows][cols rounded up to a multiple of 8]
int launch_column_sums(dbp_ctx *ctx, const void *codes, long long rows, long long cols, const float *delta_p, float *db,
                       bool beside) {
    const long long groups = (cols + 63) / 64;
    // ranges of at least 128 rows (four loads per thread), about two blocks per SM
    long long split = 2ll * ctx->sm_count / groups;
    if (split > (rows + 127) / 128) split = (rows + 127) / 128;
    if (split < 1 || groups > kMaxGroups) split = 1;
    const long long per = (rows + split - 1) / split;
    split = (rows + per - 1) / per;
    int *partials = nullptr;
    unsigned *tickets = nullptr;
    if (split > 1) {
        if (int rc = sums_workspace(ctx, static_cast<size_t>(split) * groups * 64, &partials, &tickets, &beside)) return rc;
    }
    return cuda_ok(launch_chained(column_sums_kernel, dim3(static_cast<unsigned>(groups), static_cast<unsigned>(split)), dim3(256), 0,
                                  ctx->stream, static_cast<const unsigned short *>(codes), rows, static_cast<int>(cols),
                                  (cols + 7) / 8 * 8, per, partials, tickets, delta_p, db, beside ? 1 : 0));
}

// codes: bf16 planes [B][channels][pitch] of hw codes each
int launch_plane_sums(dbp_ctx *ctx, const void *codes, long long B, long long channels, long long hw, long long pitch,
                      const float *delta_p, float *db, bool beside) {
    // ranges of at least eight planes (one per warp), about four blocks per SM
    long long split = 4ll * ctx->sm_count / channels;
    if (split > (B + 7) / 8) split = (B + 7) / 8;
    if (split < 1 || channels > kMaxGroups) split = 1;
    const long long per = (B + split - 1) / split;
    split = (B + per - 1) / per;
    int *partials = nullptr;
    unsigned *tickets = nullptr;
    if (split > 1)
        if (int rc = sums_workspace(ctx, static_cast<size_t>(split) * channels, &partials, &tickets, &beside)) return rc;
    return cuda_ok(launch_chained(plane_sums_kernel, dim3(static_cast<unsigned>(channels), static_cast<unsigned>(split)), dim3(256), 0,
                                  ctx->stream, static_cast<const unsigned short *>(codes), static_cast<int>(B), hw, pitch,
                                  static_cast<int>(per), partials, tickets, delta_p, db, beside ? 1 : 0));
}

}  // namespace dbp
