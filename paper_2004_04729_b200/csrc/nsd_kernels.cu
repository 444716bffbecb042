// NSD quantization kernels: one-pass statistics (Algorithm 1, std line), dither + quantize +
// compaction (Section 3.1, Eq. (nsd)), and expansion of the sparse structure to dense codes.
//
// Both streaming kernels are bound by HBM bandwidth: 128-bit loads of delta_z, 128-bit stores
// of the packed codes, bitmap words and offsets assembled with warp shuffles.
#include "nsd_common.cuh"

namespace dbp {

namespace {

using namespace nsd;

constexpr int kThreads = 256;
constexpr int kStatBlocksPerSM = 4, kStatUnroll = 4;       // of the statistics kernel: blocks per SM, vectors of a thread per tile

// read-once data: do not keep the line in L1
__device__ __forceinline__ uint4 load_stream(const void *p) {
    uint4 q;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(q.x), "=r"(q.y), "=r"(q.z), "=r"(q.w) : "l"(p));
    return q;
}

// ---------------------------------------------------------------- statistics (sigma, Delta)
// Sum and sum of squares of every element's distance from a pivot (the tensor's first element):
// fp32 inside one 128-bit chunk, fp64 across chunks, one pair of partial sums per block; the quantizer that follows adds
// the blocks' sums up in a fixed order (step_of, nsd_common.cuh), so the step size does not depend on scheduling. The
// variance is shift-invariant, and with the pivot inside the data's range the moments stay of the order of sigma: a
// constant tensor gives exactly 0 and a mean far from 0 costs no accuracy (raw moments would cancel).
// MASKED (fp32 only): the tensor is delta_a and the statistics are those of delta_a where mask != 0, else 0 (the
// ReLU derivative folded into the read; one byte per element).
template <bool MASKED>
__device__ __forceinline__ void mask4(const unsigned char *mask, long long e, float (&v)[4]) {
    if (MASKED) {
        const uchar4 m = __ldg(reinterpret_cast<const uchar4 *>(mask + e));
        v[0] = m.x ? v[0] : 0.f; v[1] = m.y ? v[1] : 0.f; v[2] = m.z ? v[2] : 0.f; v[3] = m.w ? v[3] : 0.f;
    }
}
template <bool MASKED>
__device__ __forceinline__ void mask4(const unsigned char *, long long, float (&)[8]) {}   // bf16 tensors take no mask

// Rows of a matrix re-written as bf16 rows of `pitch` values (a multiple of 8, the extra columns zero): bf16 rows
// copied, fp32 rows as two pieces, [rows][pitch] the rounded values and, rows * pitch further on, what the rounding
// left over, rounded again. A thread takes eight columns of one row.
// ODD: fp32 rows may start on any element; an instance of its own, because its registers keep blocks of the others out of places beside
// other kernels (38 and 32; ResNet-50 layer set 844 us in one kernel, 839 in two, 64 -> 64 fp32 at 32x32 80.7 and 79.5).
template <bool ODD>
__device__ __forceinline__ void rows_job(const RowsJob &j, long long first, long long stride) {
    const unsigned gpr = static_cast<unsigned>(j.pitch / 8);
    const long long n = j.rows * gpr, piece = j.rows * j.pitch;
    for (long long i = first; i < n; i += stride) {
        long long row;
        unsigned g;
        if ((n >> 31) == 0) {                      // 32-bit divisions cost a fraction of 64-bit ones
            row = static_cast<unsigned>(i) / gpr;
            g = static_cast<unsigned>(i) - static_cast<unsigned>(row) * gpr;
        } else {
            row = i / gpr;
            g = static_cast<unsigned>(i - row * gpr);
        }
        const long long c0 = g * 8ll, left = j.cols - c0;          // left > 0
        unsigned short *dst = static_cast<unsigned short *>(j.dst) + row * j.pitch + c0;
        if (j.f32) {
            const float *src = static_cast<const float *>(j.src) + row * j.cols + c0;
            float x[8];
            if (left >= 8 && (j.cols & 3) == 0) {
                const float4 a = __ldg(reinterpret_cast<const float4 *>(src)), b = __ldg(reinterpret_cast<const float4 *>(src + 4));
                x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
            } else {
                // rows that start anywhere: the three 16-byte words that hold the eight values, and a shift (value by value a linear layer
                // of 275 outputs of 3761 inputs, batch 31, takes 20.7 us, 19.2 so)
                const long long off = row * j.cols + c0, at = off & ~3ll;
                const int sh = static_cast<int>(off & 3);
                if (ODD && at + 12 <= j.rows * j.cols) {
                    const float4 *const p4 = reinterpret_cast<const float4 *>(static_cast<const float *>(j.src) + at);
                    const float4 a = __ldg(p4), b = __ldg(p4 + 1), c = __ldg(p4 + 2);
                    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
                    float y[9];
#pragma unroll
                    for (int e = 0; e < 9; ++e) y[e] = sh & 2 ? w[e + 2] : w[e];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = e < left ? (sh & 1 ? y[e + 1] : y[e]) : 0.f;
                } else {                               // the matrix's last values, one by one
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = e < left ? __ldg(src + e) : 0.f;
                }
            }
            unsigned h[4], l[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const __nv_bfloat162 hh = __floats2bfloat162_rn(x[2 * e], x[2 * e + 1]);
                const float2 hf = __bfloat1622float2(hh);
                const __nv_bfloat162 ll = __floats2bfloat162_rn(x[2 * e] - hf.x, x[2 * e + 1] - hf.y);
                h[e] = *reinterpret_cast<const unsigned *>(&hh);
                l[e] = *reinterpret_cast<const unsigned *>(&ll);
            }
            *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4 *>(dst + piece) = make_uint4(l[0], l[1], l[2], l[3]);
        } else {
            if (left >= 8 && (j.cols & 3) == 0) {                     // rows start on 8-byte boundaries
                const unsigned short *src8 = static_cast<const unsigned short *>(j.src) + row * j.cols + c0;
                const uint2 a = __ldg(reinterpret_cast<const uint2 *>(src8)), b = __ldg(reinterpret_cast<const uint2 *>(src8 + 4));
                *reinterpret_cast<uint4 *>(dst) = make_uint4(a.x, a.y, b.x, b.y);
                continue;
            }
            // the two 16-byte words that hold the eight values, whatever the row's start, and a shift (32-bit loads before: 59 x 344
            // rows of 59 x 59 values 65 us)
            const long long off = row * j.cols + c0, total = j.rows * j.cols, at = off & ~7ll;
            const unsigned short *src = static_cast<const unsigned short *>(j.src);
            const int sh = static_cast<int>(off & 7), nv = left < 8 ? static_cast<int>(left) : 8;
            unsigned w[4];
            if (at + 16 <= total) {
                const uint4 lo = __ldg(reinterpret_cast<const uint4 *>(src + at)), hi = __ldg(reinterpret_cast<const uint4 *>(src + at + 8));
                const unsigned x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                unsigned y[6], z[5];
#pragma unroll
                for (int e = 0; e < 6; ++e) y[e] = sh & 4 ? x[e + 2] : x[e];
#pragma unroll
                for (int e = 0; e < 5; ++e) z[e] = sh & 2 ? y[e + 1] : y[e];
#pragma unroll
                for (int e = 0; e < 4; ++e) w[e] = __funnelshift_r(z[e], z[e + 1], (sh & 1) * 16);
            } else {                               // the tensor's last values, one by one
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    w[e] = 2 * e < nv ? __ldg(src + off + 2 * e) : 0u;
                    if (2 * e + 1 < nv) w[e] |= static_cast<unsigned>(__ldg(src + off + 2 * e + 1)) << 16;
                }
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (2 * e >= nv) w[e] = 0u;
                else if (2 * e + 1 >= nv) w[e] &= 0xffffu;
            }
            *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// beside: the kernel before this one on the stream writes nothing this one reads (the quantizer, whose CTAs let this
// kernel start once they have seen everything before them complete): it works beside that kernel, whose issue slots are
// what is busy, and waits for it only before it ends, so that the kernels behind this one still come after both. For that one waiting
// block is enough, and the others leave their places to blocks that found none (fp32 rows: VGG-16 layer set 683 us with all of them
// waiting, 677 so); of bf16 rows all wait, which keeps dX's CTAs from taking the SMs in front of an earlier call's dW
// (ResNet-50 layer set 841 us, 845 with one). By the type and not by whether an earlier dW is outstanding: with nothing outstanding bf16
// calls take the same either way (160 -> 320 at 13x13, batch 64: 30.8 both), and behind a dW fp32 calls gain nothing from waiting (VGG-16
// 663, 669).
template <bool ODD>
__global__ void __launch_bounds__(kThreads) rows_job_kernel(const RowsJob j, int beside) {
    if (!beside) chain_wait();
    chain_release();
    rows_job<ODD>(j, static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x, static_cast<long long>(gridDim.x) * kThreads);
    if (beside && (blockIdx.x == 0 || !j.f32)) chain_wait();
}

// a block's sums
__device__ __forceinline__ void leave_sums(double d1, double d2, double *__restrict__ to) {
    __shared__ double sh1[kThreads / 32], sh2[kThreads / 32];
    d1 = warp_sum(d1);
    d2 = warp_sum(d2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) { sh1[warp] = d1; sh2[warp] = d2; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int w = 0; w < kThreads / 32; ++w) { a += sh1[w]; b += sh2[w]; }
        *reinterpret_cast<double2 *>(to) = make_double2(a, b);
    }
}

// PARTS: there are more parts (pairs of sums) than blocks, and a block makes several of them one after the other
// MOST: blocks of an SM that the registers have to allow
template <typename T, bool MASKED, bool PARTS = false, int MOST = kStatBlocksPerSM>
__global__ void __launch_bounds__(kThreads, MOST < kStatBlocksPerSM ? MOST : 0)
statistics_kernel(const T *__restrict__ x, long long n, int nparts, double *__restrict__ partials,
                  DeviceState *__restrict__ st, unsigned long long *__restrict__ nnz_out,
                  const unsigned char *__restrict__ mask, const SideJobs jobs) {
    constexpr int EPT = Vec<T>::V;
    const long long nvec = n / EPT;
    // whole tiles of kStatUnroll x kThreads 128-bit vectors, a block at a time, consecutive threads on consecutive vectors; the
    // next tile's loads are under way while a tile's values are added up
    constexpr int U = kStatUnroll;
    constexpr long long tile = static_cast<long long>(U) * kThreads;
    const long long ntile = nvec / tile;
    struct Batch { uint4 raw[U]; unsigned msk[MASKED ? U : 1]; } even, odd;
    auto load = [&](long long t, Batch &b) {
        const long long v0 = t * tile + threadIdx.x;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            b.raw[u] = load_stream(x + (v0 + u * kThreads) * EPT);
            if (MASKED) b.msk[u] = __ldg(reinterpret_cast<const unsigned *>(mask) + v0 + u * kThreads);
        }
    };
    chain_wait();
    chain_release();
    if (blockIdx.x < ntile) load(blockIdx.x, even);       // on its way during the side jobs
    // side job for the layer's weight-gradient kernel, which adds its partial sums into dW: clear it
    {
        const long long first = static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x, step = static_cast<long long>(gridDim.x) * kThreads;
        const long long zero_n16 = static_cast<long long>(jobs.zero_bytes / 16);
        for (long long i = first; i < zero_n16; i += step) static_cast<uint4 *>(jobs.zero)[i] = make_uint4(0u, 0u, 0u, 0u);
        if (first < static_cast<long long>(jobs.zero_bytes / 4) - 4 * zero_n16) static_cast<unsigned *>(jobs.zero)[4 * zero_n16 + first] = 0u;
        // side jobs for the layer's product kernels: operands re-written as bf16 rows the copy engine can address
        for (int j = 0; j < jobs.nrows; ++j) rows_job<true>(jobs.rows[j], first, step);
    }
    // side job for the layer's 3x3 input-gradient kernel: weights [co][ci][9] -> [tap][co][ci] bf16 (for fp32
    // weights two pieces: taps 0-8 the values rounded to bf16, taps 9-17 the remainders rounded to bf16).
    // w_phase_cin > 0: the layer is a stride-2 layer run on the four phase images of its input; w_src holds that
    // layer's own weights [co][w_phase_cin][9] and channel ph * w_phase_cin + c of the re-laid weights is phase
    // ph = 2 py + px of channel c, whose tap (ty, tx) is the strided layer's tap ky = 0 for (py, ty) = (1, 0),
    // 1 for (0, 1), 2 for (1, 1), kx likewise, and zero for every other pair.
    if (jobs.w_src != nullptr) {
        const void *w_src = jobs.w_src;
        unsigned short *w_dst = static_cast<unsigned short *>(jobs.w_dst);
        const int w_f32 = jobs.w_f32, w_cin = static_cast<int>(jobs.Cin), w_phase_cin = jobs.phase_cin;
        const int w_pitch = (w_cin + 7) & ~7;      // rows of a multiple of 16 bytes, for the copy engine
        const long long w_cout = jobs.Cout;
        const long long per_tap = w_cout * w_pitch;     // taps outermost: the copy engine takes several taps in one box
        for (long long co = blockIdx.x; co < w_cout; co += gridDim.x) {
            unsigned short *dst = w_dst + co * w_pitch;
            // A thread takes two neighbouring channels and all nine taps of them, all loads first (pairs of weights where the rows
            // allow it), then one word per tap and piece, along ci. (Of an odd number of channels the last one's word reaches into
            // the row's padding.)
            const bool paired = w_phase_cin == 0 && (w_cin & 1) == 0;
            // the bits of two channels' weights, channel c's and then channel c + 1's; even rows
            auto load_pair = [&](long long base, unsigned (&w)[18]) {
                if (w_f32) {
                    const uint2 *src = reinterpret_cast<const uint2 *>(static_cast<const float *>(w_src) + base);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const uint2 v = __ldg(src + i);
                        w[2 * i] = v.x;
                        w[2 * i + 1] = v.y;
                    }
                } else {
                    const unsigned *src = reinterpret_cast<const unsigned *>(static_cast<const unsigned short *>(w_src) + base);
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        const unsigned v = __ldg(src + i);
                        w[2 * i] = v & 0xffffu;
                        w[2 * i + 1] = v >> 16;
                    }
                }
            };
            // one word (two words: fp32's pieces) of a tap
            auto store_pair = [&](int t, int c, unsigned a, unsigned b) {
                if (w_f32) {
                    const __nv_bfloat162 hi = __floats2bfloat162_rn(__uint_as_float(a), __uint_as_float(b));
                    const float2 hf = __bfloat1622float2(hi);
                    const __nv_bfloat162 lo = __floats2bfloat162_rn(__uint_as_float(a) - hf.x, __uint_as_float(b) - hf.y);
                    *reinterpret_cast<unsigned *>(dst + t * per_tap + c) = *reinterpret_cast<const unsigned *>(&hi);
                    *reinterpret_cast<unsigned *>(dst + (9 + t) * per_tap + c) = *reinterpret_cast<const unsigned *>(&lo);
                } else {
                    *reinterpret_cast<unsigned *>(dst + t * per_tap + c) = a | b << 16;
                }
            };
            if (w_phase_cin > 0 && (w_phase_cin & 1) == 0) {
                // Two channels of the strided layer with all four of their phases: its weights are read once (phase by phase, tap
                // by tap, 512 -> 512 took this kernel 16 us instead of 9)
                for (int c = 2 * threadIdx.x; c < w_phase_cin; c += 2 * kThreads) {
                    unsigned w[18];
                    load_pair((co * w_phase_cin + c) * 9, w);
#pragma unroll
                    for (int ph = 0; ph < 4; ++ph)
#pragma unroll
                        for (int t = 0; t < 9; ++t) {
                            const int ty = t / 3, tx = t % 3;
                            const int ky = (ph & 2) ? (ty == 0 ? 0 : (ty == 1 ? 2 : -1)) : (ty == 1 ? 1 : -1);
                            const int kx = (ph & 1) ? (tx == 0 ? 0 : (tx == 1 ? 2 : -1)) : (tx == 1 ? 1 : -1);
                            if (ky >= 0 && kx >= 0) store_pair(t, ph * w_phase_cin + c, w[ky * 3 + kx], w[9 + ky * 3 + kx]);
                            else if (!jobs.skip_dead) store_pair(t, ph * w_phase_cin + c, 0u, 0u);
                        }
                }
                continue;
            }
            for (int c0 = 2 * threadIdx.x; c0 < w_cin; c0 += 2 * kThreads) {
                unsigned w[18];                                        // the bits of the weights: channel c0's, then channel c0 + 1's
                if (paired) {
                    load_pair((co * w_cin + c0) * 9, w);
                } else {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int ci = c0 + h;
                        int ph = 0;
                        long long base = (co * w_cin + ci) * 9;
                        if (w_phase_cin > 0) {
                            ph = ci / w_phase_cin;
                            base = (co * w_phase_cin + (ci - ph * w_phase_cin)) * 9;
                        }
#pragma unroll
                        for (int t = 0; t < 9; ++t) {
                            const int ty = t / 3, tx = t % 3;
                            int k = t;                                 // source tap
                            bool live = true;
                            if (w_phase_cin > 0) {
                                const int ky = (ph & 2) ? (ty == 0 ? 0 : (ty == 1 ? 2 : -1)) : (ty == 1 ? 1 : -1);
                                const int kx = (ph & 1) ? (tx == 0 ? 0 : (tx == 1 ? 2 : -1)) : (tx == 1 ? 1 : -1);
                                live = ky >= 0 && kx >= 0;
                                k = ky * 3 + kx;
                            }
                            w[9 * h + t] = 0u;
                            if (live && ci < w_cin)
                                w[9 * h + t] = w_f32 ? __float_as_uint(__ldg(static_cast<const float *>(w_src) + base + k))
                                                     : static_cast<unsigned>(__ldg(static_cast<const unsigned short *>(w_src) + base + k));
                        }
                    }
                }
#pragma unroll
                for (int t = 0; t < 9; ++t) store_pair(t, c0, w[t], w[9 + t]);
            }
        }
    }
    double d1 = 0.0, d2 = 0.0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {      // the quantizer counts into these
        st->nnz = 0ull;
        if (nnz_out) *nnz_out = 0ull;
    }
    const float pivot = (!MASKED || __ldg(mask)) ? Vec<T>::one(x) : 0.f;
    const int parts = PARTS ? nparts : static_cast<int>(gridDim.x);
    const long long stride = static_cast<long long>(parts) * kThreads;
    auto add = [&](const Batch &b) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float v[EPT];
            Vec<T>::values(b.raw[u], v);
            if (MASKED) {
#pragma unroll
                for (int j = 0; j < EPT; ++j) v[j] = b.msk[u] >> (8 * j & 31) & 0xffu ? v[j] : 0.f;
            }
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int j = 0; j < EPT; ++j) {
                const float c = v[j] - pivot;
                s1 += c;
                s2 = fmaf(c, c, s2);
            }
            d1 += static_cast<double>(s1);
            d2 += static_cast<double>(s2);
        }
    };
    for (int part = blockIdx.x;;) {
        for (long long t = part; t < ntile; t += 2 * parts) {
            const long long t1 = t + parts, t2 = t1 + parts;
            if (t1 < ntile) load(t1, odd);
            add(even);
            if (t2 < ntile) load(t2, even);
            if (t1 < ntile) add(odd);
        }
        // the vectors after the last whole tile
        long long i = ntile * tile + static_cast<long long>(part) * kThreads + threadIdx.x;
        for (; i < nvec; i += stride) {
            float v[EPT];
            Vec<T>::values(Vec<T>::raw(x + i * EPT), v);
            mask4<MASKED>(mask, i * EPT, v);
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int j = 0; j < EPT; ++j) {
                const float c = v[j] - pivot;
                s1 += c;
                s2 = fmaf(c, c, s2);
            }
            d1 += static_cast<double>(s1);
            d2 += static_cast<double>(s2);
        }
        if (part == 0 && threadIdx.x == 0) {
            for (long long i = nvec * EPT; i < n; ++i) {
                const float xi = (!MASKED || __ldg(mask + i)) ? Vec<T>::one(x + i) : 0.f;
                const double c = static_cast<double>(xi) - static_cast<double>(pivot);
                d1 += c;
                d2 += c * c;
            }
        }
        leave_sums(d1, d2, partials + 2 * part);
        part += gridDim.x;
        if (!PARTS || part >= parts) break;
        __syncthreads();                             // (the sums have been read)
        if (part < ntile) load(part, even);
        d1 = d2 = 0.0;
    }
}

// The statistics of a gradient that comes out of a 2x2 max-pool's routing, written on the way (one launch and one pass less than
// the routing by itself and then statistics_kernel; LeNet-5-like chain, batch 128: 48.3 us, 42.4). A thread takes two windows of a row,
// whose elements are two vectors of four; sums as there.
template <bool MASKED>
__global__ void __launch_bounds__(kThreads)
statistics_pool_kernel(const PoolRouting pool, long long n2, double *__restrict__ partials, DeviceState *__restrict__ st,
                       unsigned long long *__restrict__ nnz_out, const unsigned char *__restrict__ mask, const SideJobs jobs) {
    chain_wait();
    chain_release();
    const long long first = static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x, step = static_cast<long long>(gridDim.x) * kThreads;
    const long long zero_n16 = static_cast<long long>(jobs.zero_bytes / 16);
    for (long long i = first; i < zero_n16; i += step) static_cast<uint4 *>(jobs.zero)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (first < static_cast<long long>(jobs.zero_bytes / 4) - 4 * zero_n16) static_cast<unsigned *>(jobs.zero)[4 * zero_n16 + first] = 0u;
    if (first == 0) {                               // the quantizer counts into these
        st->nnz = 0ull;
        if (nnz_out) *nnz_out = 0ull;
    }
    const float pivot = __ldg(pool.argmax) == 0 && (!MASKED || __ldg(mask)) ? __ldg(pool.g) : 0.f;
    const int w2 = pool.w / 2;
    double d1 = 0.0, d2 = 0.0;
    for (long long i = first; i < n2; i += step) {
        const float2 g = __ldg(reinterpret_cast<const float2 *>(pool.g) + i);
        const char2 a = __ldg(reinterpret_cast<const char2 *>(pool.argmax) + i);
        const long long row = (n2 >> 31) == 0 ? static_cast<unsigned>(i) / static_cast<unsigned>(w2) : i / w2;
        // row (plane, y) of windows starts at element row * 4 w of the output, two rows of 2 w
        const long long e = row * 4 * pool.w + (i - row * w2) * 4;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            float v[4] = {a.x == 2 * half ? g.x : 0.f, a.x == 2 * half + 1 ? g.x : 0.f, a.y == 2 * half ? g.y : 0.f, a.y == 2 * half + 1 ? g.y : 0.f};
            const long long at = e + half * 2 * pool.w;
            *reinterpret_cast<float4 *>(pool.out + at) = make_float4(v[0], v[1], v[2], v[3]);
            mask4<MASKED>(mask, at, v);
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float c = v[j] - pivot;
                s1 += c;
                s2 = fmaf(c, c, s2);
            }
            d1 += static_cast<double>(s1);
            d2 += static_cast<double>(s2);
        }
    }
    leave_sums(d1, d2, partials + 2 * blockIdx.x);
}

// A given step size: no statistics; the counters the quantizer adds to are cleared.
__global__ void clear_counts_kernel(DeviceState *st, unsigned long long *nnz_out) {
    chain_wait();
    chain_release();
    st->nnz = 0ull;
    if (nnz_out) *nnz_out = 0ull;
}

// ---------------------------------------------------------------- dither + quantize + compact
// One warp owns one 1024-element segment at a time, one lane 32 consecutive elements of it: one bitmap word, so a word
// and its popcount need no exchange between lanes, and one scan per segment gives every word's offset. The codes of a
// lane are dumped to shared memory as bytes and the non-zero ones are picked out by walking the word's bits (a few per
// lane at the sparsities this is used at); the segment leaves as coalesced stores of the 32 words, the 32 offsets and
// the packed codes. A segment that ends the tensor or holds a code out of range is decided again element by element, so that
// the others have no branch per vector (but not in a small tensor, where that is all there is: 9.8 against 8.5 us): 26 instructions an element (16 of them the decision) against 31, the call of 12.8 M bf16
// elements with its decoding 29.5 us against 31.1.
constexpr int kLanePitch = 36;                    // bytes between two lanes' codes: an odd number of words

template <typename T>
__global__ void __launch_bounds__(kThreads)
quantize_kernel(const T *__restrict__ x, long long n, unsigned long long seed, const StepSource step,
                uint32_t *__restrict__ bitmap, uint16_t *__restrict__ offsets, int8_t *__restrict__ values,
                int8_t *__restrict__ dense, DeviceState *__restrict__ st, unsigned long long *__restrict__ nnz_out) {
    constexpr int V = Vec<T>::V;
    constexpr int NV = 32 / V;                                       // vectors per lane and segment
    __shared__ __align__(16) unsigned char stage[kThreads / 32][kSegment];
    __shared__ __align__(16) unsigned char byte_s[kThreads / 32][32 * kLanePitch];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long nseg = (n + kSegment - 1) / kSegment, whole = n / kSegment;
    const long long nwarps = static_cast<long long>(gridDim.x) * (kThreads / 32);
    long long seg = static_cast<long long>(blockIdx.x) * (kThreads / 32) + warp;
    unsigned long long z = counter_of(seg * kSegment + lane * 32, seed);
    const unsigned long long stride_z = static_cast<unsigned long long>(nwarps) * (kSegment / 2) * kGamma;
    uint4 raw[NV];
    auto load = [&](long long sg) {
        if (sg >= whole) return;
        const T *src = x + sg * kSegment + lane * 32;
#pragma unroll
        for (int i = 0; i < NV; ++i) raw[i] = Vec<T>::raw(src + i * V);
    };
    load(seg);
    // A warp's first segment may be the one that ends the tensor (of a small one; later in the loop it is read element by element)
    bool ready = seg < nseg;
    if (ready && seg >= whole) {
        const long long e = seg * kSegment + lane * 32;
#pragma unroll
        for (int i = 0; i < NV; ++i)
            raw[i] = e + i * V + V <= n ? Vec<T>::raw(x + e + i * V) : load_edge(x + e + i * V, n - e - i * V);      // beyond the end: code 0
    }
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned nnz = 0, sat = 0;
    unsigned *const mine = reinterpret_cast<unsigned *>(byte_s[warp] + lane * kLanePitch);
    // one bit per non-zero byte: bit 7 of each byte, gathered by a multiplication
    auto bits_of = [](unsigned b) { return (((((b & 0x7f7f7f7fu) + 0x7f7f7f7fu) | b) & 0x80808080u) >> 7) * 0x01020408u >> 24; };
    for (; seg < nseg; seg += nwarps) {
        const long long e0 = seg * kSegment + lane * 32;
        unsigned word = 0, top = 0u;
        if (ready) {
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                float v[V];
                unsigned h[V / 2], m[V], b[V / 4];
                unsigned long long u[V / 2];
                Vec<T>::values(raw[i], v);
                dithers_at<V>(z + static_cast<unsigned long long>(i * V / 2) * kGamma, u);
                quick_codes<V>(v, u, inv, h, m, top);
                low_bytes<V>(m, b);
#pragma unroll
                for (int w = 0; w < V / 4; ++w) {
                    mine[i * (V / 4) + w] = b[w];
                    word |= bits_of(b[w]) << (i * V + 4 * w);
                }
            }
        }
        z += stride_z;
        load(seg + nwarps);
        if (!ready || needs_care(top)) {                             // the tensor's end; rare: clip, count, NaN
            word = 0;
#pragma unroll 1
            for (int w = 0; w < 8; ++w) {
                unsigned long long u[2];
                dithers_of<4>(e0 + 4 * w, seed, u);
                unsigned b = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const long long e = e0 + 4 * w + j;
                    float ua, ub;
                    unpack2(u[j >> 1], ua, ub);
                    if (e < n) b |= (careful_bits(Vec<T>::one(x + e), inv, (j & 1) ? ub : ua, sat) & 0xffu) << (8 * j);
                }
                mine[w] = b;
                word |= bits_of(b) << (4 * w);
            }
        }
        const unsigned pc = __popc(word);
        unsigned incl = pc;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned up = __shfl_up_sync(kFull, incl, o);
            if (lane >= o) incl += up;
        }
        const unsigned total = __shfl_sync(kFull, incl, 31);
        bitmap[seg * kWordsPerSegment + lane] = word;
        offsets[seg * kWordsPerSegment + lane] = static_cast<uint16_t>(incl - pc);
        if (dense != nullptr) {
            if (e0 + 32 <= n) {
                reinterpret_cast<uint4 *>(dense + e0)[0] = make_uint4(mine[0], mine[1], mine[2], mine[3]);
                reinterpret_cast<uint4 *>(dense + e0)[1] = make_uint4(mine[4], mine[5], mine[6], mine[7]);
            } else {
                for (int j = 0; j < 32; ++j)
                    if (e0 + j < n) dense[e0 + j] = static_cast<int8_t>(reinterpret_cast<const unsigned char *>(mine)[j]);
            }
        }
        unsigned char *dst = stage[warp] + (incl - pc);
        const unsigned char *src = reinterpret_cast<const unsigned char *>(mine);
        for (unsigned m = word; m; m &= m - 1) *dst++ = src[__ffs(m) - 1];
        __syncwarp();
        for (unsigned i = lane * 16; i < total; i += 512)
            *reinterpret_cast<uint4 *>(values + seg * kSegment + i) = *reinterpret_cast<const uint4 *>(&stage[warp][i]);
        __syncwarp();
        nnz += lane == 0 ? total : 0u;
        ready = seg + nwarps < whole;
    }
    publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nnz_out);
}

// One warp per segment, one lane per bitmap word. The segment's packed codes come in as whole lines; a lane takes its
// word four bits at a time: the next codes (a 32-bit window at the running rank, from two words of shared memory) are
// spread to the bytes whose bits are set by one byte permutation, whose selector for the sixteen patterns is a table.
__global__ void __launch_bounds__(kThreads)
decode_kernel(const uint32_t *__restrict__ bitmap, const uint16_t *__restrict__ offsets,
              const int8_t *__restrict__ values, long long n, int8_t *__restrict__ dense) {
    __shared__ __align__(16) unsigned char stage[kThreads / 32][kSegment + 16];
    __shared__ unsigned sel_s[16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 16) {
        unsigned sel = 0, r = 0;
        for (int b = 0; b < 4; ++b) sel |= ((threadIdx.x >> b) & 1 ? r++ : 4u) << (4 * b);      // selector 4: a zero byte
        sel_s[threadIdx.x] = sel;
    }
    __syncthreads();
    chain_wait();
    chain_release();
    const long long nseg = (n + kSegment - 1) / kSegment;
    const long long nwarps = static_cast<long long>(gridDim.x) * (kThreads / 32);
    for (long long seg = static_cast<long long>(blockIdx.x) * (kThreads / 32) + warp; seg < nseg; seg += nwarps) {
        const long long w = seg * kWordsPerSegment + lane;
        const unsigned word = __ldcg(bitmap + w), off = __ldcg(offsets + w);
        // a first line is on its way with the words: at the usual sparsities the segment has few more
        uint4 *line = reinterpret_cast<uint4 *>(stage[warp]);
        const uint4 *src = reinterpret_cast<const uint4 *>(values + seg * kSegment);
        if (lane < 8) line[lane] = __ldcg(src + lane);
        const unsigned total = __shfl_sync(kFull, off + __popc(word), 31);
        for (unsigned i = lane + 8; i * 16 < total; i += 32) line[i] = __ldcg(src + i);
        __syncwarp();
        const unsigned *codes = reinterpret_cast<const unsigned *>(stage[warp]);
        unsigned pk[8], r = off;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            const unsigned m = (word >> (4 * g)) & 15u;
            const unsigned win = __funnelshift_r(codes[r >> 2], codes[(r >> 2) + 1], 8 * (r & 3));
            pk[g] = __byte_perm(win, 0u, sel_s[m]);
            r += __popc(m);
        }
        __syncwarp();
        const long long e0 = w * 32;
        if (e0 + 32 <= n) {
            uint4 *dst = reinterpret_cast<uint4 *>(dense + e0);
            dst[0] = make_uint4(pk[0], pk[1], pk[2], pk[3]);
            dst[1] = make_uint4(pk[4], pk[5], pk[6], pk[7]);
        } else {
            for (int j = 0; j < 32; ++j)
                if (e0 + j < n) dense[e0 + j] = static_cast<int8_t>((pk[j >> 2] >> (8 * (j & 3))) & 0xff);
        }
    }
}

}  // namespace


int launch_rows_job(dbp_ctx *ctx, const RowsJob &job, bool beside) {
    long long b = (job.rows * (job.pitch / 8) + kThreads - 1) / kThreads;
    if (b > static_cast<long long>(ctx->sm_count) * 8) b = static_cast<long long>(ctx->sm_count) * 8;
    const bool odd = job.f32 && (job.cols & 3) != 0;
    return cuda_ok(launch_chained(odd ? rows_job_kernel<true> : rows_job_kernel<false>, dim3(static_cast<unsigned>(b)), dim3(kThreads), 0, ctx->stream, job, beside ? 1 : 0));
}

int launch_statistics(dbp_ctx *ctx, const void *delta, int dtype, long long numel, float scale,
                      const float *delta_in, float *const (&publish)[2], unsigned long long *nnz_out, StepSource *step,
                      const SideJobs &jobs, const uint8_t *mask) {
    if (mask != nullptr && dtype != DBP_F32) return DBP_EUNSUPPORTED;
    step->publish[0] = &ctx->state->delta;
    step->publish[1] = publish[0];
    step->publish[2] = publish[1];
    if (!(scale > 0.f)) {      // the step size is given: no statistics kernel, so no side jobs either (the caller sees to the weights)
        if (jobs.zero && cudaMemsetAsync(jobs.zero, 0, jobs.zero_bytes, ctx->stream) != cudaSuccess) return fail_cuda("clearing dW");
        for (int j = 0; j < jobs.nrows; ++j)
            if (int rc = launch_rows_job(ctx, jobs.rows[j], false)) return rc;
        step->given = delta_in;
        return cuda_ok(launch_chained(clear_counts_kernel, dim3(1), dim3(1), 0, ctx->stream, ctx->state, nnz_out));
    }
    const bool routed = jobs.pool.g != nullptr;
    const int ept = dtype == DBP_F32 ? 4 : 8;
    long long blocks = numel / ept / (kThreads * kStatUnroll);          // one block per tile
    if (routed) blocks = (numel / 8 + kThreads - 1) / kThreads;      // one pair of windows per thread
    if (blocks < 1) blocks = 1;
    // the side jobs want blocks of their own when the tensor is small (a block beyond the tensor's tiles adds zeros)
    if (jobs.w_src != nullptr && blocks < jobs.Cout) blocks = jobs.Cout;
    if (jobs.zero != nullptr && blocks < static_cast<long long>(jobs.zero_bytes / (16 * kThreads * 4))) blocks = static_cast<long long>(jobs.zero_bytes / (16 * kThreads * 4));
    for (int j = 0; j < jobs.nrows; ++j) {         // two eight-column groups per thread
        const long long b = jobs.rows[j].rows * (jobs.rows[j].pitch / 8) / (2 * kThreads);
        if (blocks < b) blocks = b;
    }
    if (blocks > ctx->partial_blocks) blocks = ctx->partial_blocks;
    // Four resident blocks per SM, each walking its tiles of four vectors a thread with the next tile's loads under way (two blocks,
    // eight vectors, one tile's loads at a time before: ResNet-50 layer set 845 us against 839, VGG-16 762 against 756, 2048 -> 1000 at
    // batch 256 23.6 against 23.1, the largest tensors the same: 103 MB in 16 us). Two, three or six blocks with this kernel: 853, 847,
    // 847. The weight re-laying side job wants one block per output channel.
    if (jobs.w_src == nullptr && blocks > static_cast<long long>(ctx->sm_count) * kStatBlocksPerSM)
        blocks = static_cast<long long>(ctx->sm_count) * kStatBlocksPerSM;
    // Beside an earlier call's dW, whose CTAs leave the registers for two of them, four blocks ran two after two, and the quantizer came to
    // its loads and dithers only when the last ones had started. fp32 tensors of 100 MB and more are taken by two blocks per SM there, two
    // parts each (the sums are the same: the step size does not depend on what is beside): 1x1 64 -> 256 at 56x56, batch 64, overlapped
    // 176 us, 166 so; 128 -> 512 at 28x28 (103 MB) 93.1, 88.0. Smaller ones wait for memory's latency then: 300 -> 200 at 30x31, batch 100
    // (74 MB), 206, 211; bf16 tensors too (ResNet-50 set 840, 855).
    const bool halved = dtype == DBP_F32 && numel >= 25000000 && ctx->aux_pending && blocks > 2ll * ctx->sm_count;
    const long long grid = halved ? 2ll * ctx->sm_count : blocks;
    auto go = [&](auto kern, auto x, const unsigned char *m) {
        return launch_chained(kern, dim3(static_cast<unsigned>(grid)), dim3(kThreads), 0, ctx->stream, x, numel, static_cast<int>(blocks),
                              ctx->partials, ctx->state, nnz_out, m, jobs);
    };
    step->partials = ctx->partials;
    step->nparts = static_cast<int>(blocks);
    step->inv_numel = 1.0 / static_cast<double>(numel);
    step->scale = scale;
    const unsigned char *m = static_cast<const unsigned char *>(mask);
    if (routed) {
        step->late = 1;
        return cuda_ok(launch_chained(m != nullptr ? statistics_pool_kernel<true> : statistics_pool_kernel<false>, dim3(static_cast<unsigned>(blocks)),
                                      dim3(kThreads), 0, ctx->stream, jobs.pool, numel / 8, ctx->partials, ctx->state, nnz_out, m, jobs));
    }
    const float *xf = static_cast<const float *>(delta);
    // Side jobs that are more than a store or a pair of loads at a time (rows re-written, 3x3 weights of an odd channel count), in a grid of
    // two blocks per SM at most with nothing beside it: the instance with up to 128 registers keeps more of their loads under way than the
    // 64 that four blocks leave. us with 64, with more: fp32 1000 -> 999 of 777, batch 1000, 32.6, 30.6; 384 of 1496, batch 327, 16.3, 15.2;
    // 3x3 961 -> 224 at 14x15, batch 8, dX alone 42.2, 37.7; bf16 999 of 777 25.6, 24.8. Other calls lose by it, because the quantizer's blocks
    // find no registers beside these (ResNet-50 set of 16 images 406.4, 410.3; in every grid, 64 images: 836, 850).
    const __nv_bfloat16 *xb = static_cast<const __nv_bfloat16 *>(delta);
    const bool odd_weights = jobs.w_src != nullptr && ((jobs.phase_cin > 0 ? jobs.phase_cin : jobs.Cin) & 1) != 0;
    const bool few = (jobs.nrows > 0 || odd_weights) && grid <= 2ll * ctx->sm_count && !ctx->aux_pending;
    const cudaError_t e = few ? (dtype != DBP_F32 ? go(statistics_kernel<__nv_bfloat16, false, false, 2>, xb, m)
                                 : mask != nullptr ? go(statistics_kernel<float, true, false, 2>, xf, m)
                                                   : go(statistics_kernel<float, false, false, 2>, xf, m))
                          : dtype != DBP_F32 ? go(statistics_kernel<__nv_bfloat16, false>, xb, m)
                          : mask != nullptr ? (halved ? go(statistics_kernel<float, true, true>, xf, m) : go(statistics_kernel<float, true>, xf, m))
                                            : (halved ? go(statistics_kernel<float, false, true>, xf, m) : go(statistics_kernel<float, false>, xf, m));
    return cuda_ok(e);
}

int launch_quantize(dbp_ctx *ctx, const void *delta, int dtype, long long numel,
                    unsigned long long seed, const StepSource &step, uint32_t *bitmap,
                    uint16_t *offsets, int8_t *values, int8_t *dense,
                    unsigned long long *nnz_out) {
    const long long nseg = (numel + kSegment - 1) / kSegment;
    long long blocks = (nseg + kThreads / 32 - 1) / (kThreads / 32);
    const long long cap = static_cast<long long>(ctx->sm_count) * 4;
    if (blocks > cap) blocks = cap;
    auto go = [&](auto kern, auto x) {
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream, x, numel, seed, step,
                                      bitmap, offsets, values, dense, ctx->state, nnz_out));
    };
    return dtype == DBP_F32 ? go(quantize_kernel<float>, static_cast<const float *>(delta))
                            : go(quantize_kernel<__nv_bfloat16>, static_cast<const __nv_bfloat16 *>(delta));
}

int launch_decode(dbp_ctx *ctx, const uint32_t *bitmap, const uint16_t *offsets,
                  const int8_t *values, long long numel, int8_t *dense) {
    const long long nseg = (numel + kSegment - 1) / kSegment;
    long long blocks = (nseg + kThreads / 32 - 1) / (kThreads / 32);
    const long long cap = static_cast<long long>(ctx->sm_count) * 8;
    if (blocks > cap) blocks = cap;
    return cuda_ok(launch_chained(decode_kernel, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream, bitmap,
                                  offsets, values, numel, dense));
}

}  // namespace dbp
