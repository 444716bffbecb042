// NSD quantization for the product kernels (Section 3.1, Eq. (nsd)): the same codes as quantize_kernel, written only as
// the dense arrays the dX / dW kernels read, without the bitmap / offsets / packed-values structure. Used when the caller
// did not ask for the sparse structure, so the pass costs one read of delta_z and one write of the codes.
//
// What bounds the kernels are instructions: 32 per element of a bf16 tensor (52 for planes of odd sizes), 13 of them the
// SplitMix64 draw, at 66 % of the issue slots (56 %; 24 warps per SM, which wait for the ALU pipe, for fixed latencies and for
// their turn) and 0.2 of the memory bandwidth. 12.8 M elements: 22 us, and 16 with the draw left out. So the arithmetic works
// on pairs (nsd_common.cuh). A thread's first vectors of delta_z and their dithers need
// nothing of the statistics kernel that runs before: they are loaded and drawn before the wait for it. That is safe
// because the statistics kernel lets this one start only once all of its own blocks have seen the kernels before it
// complete. In the loop the next vectors are loaded before the current ones are stored.
#include "nsd_common.cuh"

namespace dbp {

namespace {

using namespace nsd;

constexpr int kThreads = 256;
constexpr int kBlocksPerSM = 3;                   // resident blocks the dense quantizer is compiled for

// Where the codes go. dense8: one byte per element, same order as delta_z (may be null).
// planes16: bf16 codes as [plane][pitch] with plane = e / hw (may be null); the pitch is a
// multiple of 8 so that every plane starts on a 16-byte boundary.
struct CodeSinks {
    int8_t *dense8;
    unsigned short *planes16;
    long long hw, pitch;
    int count;                    // add nnz / clipped counts to the context's counters
};

// plane = e / hw and the offset inside it; a 32-bit division when the index allows it (a 64-bit
// one costs several times as many instructions)
__device__ __forceinline__ void split_index(long long e, long long hw, long long &plane, long long &pp) {
    if (((e | hw) >> 32) == 0) {
        const unsigned q = static_cast<unsigned>(e) / static_cast<unsigned>(hw);
        plane = q;
        pp = static_cast<unsigned>(e) - q * static_cast<unsigned>(hw);
    } else {
        plane = e / hw;
        pp = e - plane * hw;
    }
}

// f: the codes as floats, h: as packed bf16
template <int V>
__device__ __forceinline__ void store_codes(const CodeSinks &o, long long e0, const float (&f)[V], const unsigned (&h)[V / 2]) {
    if (o.dense8 != nullptr) {
        unsigned pk[V / 4];
        pack_bytes<V>(f, pk);
        if (V == 4) *reinterpret_cast<unsigned *>(o.dense8 + e0) = pk[0];
        else *reinterpret_cast<uint2 *>(o.dense8 + e0) = make_uint2(pk[0], pk[V / 4 - 1]);
    }
    if (o.planes16 != nullptr) {
        if (o.pitch == o.hw) {                      // planes are back to back: same order as delta_z
            if (V == 4) *reinterpret_cast<uint2 *>(o.planes16 + e0) = make_uint2(h[0], h[1]);
            else *reinterpret_cast<uint4 *>(o.planes16 + e0) = make_uint4(h[0], h[1], h[V / 2 - 2], h[V / 2 - 1]);
        } else if ((o.hw & 3) == 0) {
            // e0 and the plane size are multiples of 4: each group of four codes lies in one plane
            // and starts on an 8-byte boundary there
            long long plane, pp;
            split_index(e0, o.hw, plane, pp);
#pragma unroll
            for (int g = 0; g < V / 4; ++g) {
                *reinterpret_cast<uint2 *>(o.planes16 + plane * o.pitch + pp) = make_uint2(h[2 * g], h[2 * g + 1]);
                pp += 4;
                if (pp == o.hw) { pp = 0; ++plane; }
            }
        } else {
            // odd plane sizes: code by code, or two at a time where the pair starts on an even offset
            // of its plane and does not run over the plane's end
            long long plane, pp;
            split_index(e0, o.hw, plane, pp);
            unsigned short *dst = o.planes16 + plane * o.pitch + pp;
            long long left = o.hw - pp;                           // codes until the plane ends
            const long long gap = o.pitch - o.hw;
#pragma unroll
            for (int j = 0; j < V; j += 2) {
                if (left >= 2 && (reinterpret_cast<uintptr_t>(dst) & 3) == 0) {
                    *reinterpret_cast<unsigned *>(dst) = h[j >> 1];
                    dst += 2;
                    left -= 2;
                    if (left == 0) { left = o.hw; dst += gap; }
                } else {
                    *dst++ = static_cast<unsigned short>(h[j >> 1]);
                    if (--left == 0) { left = o.hw; dst += gap; }
                    *dst++ = static_cast<unsigned short>(h[j >> 1] >> 16);
                    if (--left == 0) { left = o.hw; dst += gap; }
                }
            }
        }
    }
}
__device__ __forceinline__ void store_code(const CodeSinks &o, long long e, unsigned byte) {
    if (o.dense8 != nullptr) o.dense8[e] = static_cast<int8_t>(byte);
    if (o.planes16 != nullptr) {
        const long long plane = e / o.hw;
        const float f = static_cast<float>(static_cast<int>(static_cast<signed char>(byte)));
        o.planes16[plane * o.pitch + (e - plane * o.hw)] = static_cast<unsigned short>(__float_as_uint(f) >> 16);
    }
}

// mask (fp32 tensors only): x is delta_a and the gradient is delta_a where mask != 0, else 0. The four mask bytes of a
// vector as one word.
__device__ __forceinline__ unsigned mask_word(const unsigned char *mask, long long e) { return __ldg(reinterpret_cast<const unsigned *>(mask + e)); }
__device__ __forceinline__ void apply_mask(unsigned m, float (&v)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (m >> (8 * j)) & 0xffu ? v[j] : 0.f;
}
__device__ __forceinline__ void apply_mask(unsigned, float (&)[8]) {}                 // bf16 tensors take no mask

template <typename T, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_dense_kernel(const T *__restrict__ x, long long n, unsigned long long seed, const StepSource step,
                      const CodeSinks out, DeviceState *__restrict__ st, const unsigned char *__restrict__ mask) {
    constexpr int V = Vec<T>::V;
    const long long nvec = n / V;
    const long long stride = static_cast<long long>(gridDim.x) * kThreads;
    long long i = static_cast<long long>(blockIdx.x) * kThreads + threadIdx.x;
    // two vectors per thread and round: i and i + stride
    uint4 r0, r1;
    unsigned m0 = 0, m1 = 0;
    unsigned long long u0[V / 2], u1[V / 2];
    auto load = [&](long long k) {
        r0 = k < nvec ? Vec<T>::raw(x + k * V) : make_uint4(0u, 0u, 0u, 0u);
        r1 = k + stride < nvec ? Vec<T>::raw(x + (k + stride) * V) : make_uint4(0u, 0u, 0u, 0u);
        if (MASKED) {
            m0 = k < nvec ? mask_word(mask, k * V) : 0u;
            m1 = k + stride < nvec ? mask_word(mask, (k + stride) * V) : 0u;
        }
    };
    auto draw = [&](long long k) {
        dithers_of<V>(k * V, seed, u0);
        dithers_of<V>((k + stride) * V, seed, u1);
    };
    load(i);
    draw(i);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(step, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: x * 0 + u < 1, every code 0 (NaN too)
    unsigned sat = 0, nz2 = 0, nnz = 0;
    for (; i < nvec; ) {
        float v[V], f0[V], f1[V];
        Vec<T>::values(r0, v);
        if (MASKED) apply_mask(m0, v);
        decide<V>(v, u0, inv, f0, sat);
        Vec<T>::values(r1, v);
        if (MASKED) apply_mask(m1, v);
        const bool two = i + stride < nvec;
        decide<V>(v, u1, inv, f1, sat);
        const long long k = i;
        i += 2 * stride;
        load(i);
        unsigned h0[V / 2], h1[V / 2];
        pack_bf16<V>(f0, h0);
        pack_bf16<V>(f1, h1);
        count_pairs<V>(h0, nz2);
        store_codes<V>(out, k * V, f0, h0);
        if (two) {
            count_pairs<V>(h1, nz2);
            store_codes<V>(out, (k + stride) * V, f1, h1);
        }
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
        if (i < nvec) draw(i);
    }
    nnz += pairs_total(nz2);
    if (blockIdx.x == 0 && threadIdx.x == 0) {      // the n % V last elements, one by one
        for (long long e = nvec * V; e < n; ++e) {
            float ua, ub;
            unpack2(dither2(counter_of(e & ~1ll, seed)), ua, ub);
            const unsigned q = careful_bits(!MASKED || __ldg(mask + e) ? Vec<T>::one(x + e) : 0.f, inv, (e & 1) ? ub : ua, sat) & 0xffu;
            store_code(out, e, q);
            nnz += q != 0u;
        }
    }
    if (out.count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}


// ---------------------------------------------------------------- position-major bf16 codes
// The same codes, written as bf16 in the order [image][position][channel] (the 3x3 tensor-core
// kernels read this form: a row of 64 channels of one position is 128 contiguous bytes, so a
// rectangular patch of positions with its halo is one tiled copy and a tap of the filter is a row
// offset inside it). delta_z itself is [image][channel][position], so a block transposes tiles of
// 64 channels x 64 positions through shared memory: rows of the input are read along the
// positions, rows of the output are written along the channels. The dither of an element is
// still keyed on its index in delta_z's own order.
constexpr int kTC = 64, kTP = 64;                 // channels x positions per tile
constexpr int kTileBytes = kTP * kTC * 2;

// shared-memory byte offset of (position p, channel c) inside a tile: 128-byte rows, the
// 16-byte pieces of a row permuted by the row's group of eight
__device__ __forceinline__ unsigned tile_off(int p, int c) {
    return static_cast<unsigned>(p) * 128u + (((static_cast<unsigned>(c) >> 3) ^ ((static_cast<unsigned>(p) >> 3) & 7u)) << 4) +
           ((static_cast<unsigned>(c) & 7u) << 1);
}

// V of the elements of a 128-bit vector (8-byte loads for bf16 planes that are only a multiple of 4)
template <typename T, int V>
__device__ __forceinline__ uint4 load_raw(const T *p) {
    if (sizeof(T) * V == 16) return __ldg(reinterpret_cast<const uint4 *>(p));
    const uint2 q = __ldg(reinterpret_cast<const uint2 *>(p));
    return make_uint4(q.x, q.y, 0u, 0u);
}
__device__ __forceinline__ void values_of(const float *, const uint4 &q, float (&v)[4]) { Vec<float>::values(q, v); }
__device__ __forceinline__ void values_of(const __nv_bfloat16 *, const uint4 &q, float (&v)[8]) { Vec<__nv_bfloat16>::values(q, v); }
__device__ __forceinline__ void values_of(const __nv_bfloat16 *, const uint4 &q, float (&v)[4]) {
    v[0] = __uint_as_float(q.x << 16); v[1] = __uint_as_float(q.x & 0xffff0000u);
    v[2] = __uint_as_float(q.y << 16); v[3] = __uint_as_float(q.y & 0xffff0000u);
}

template <int V>
__device__ __forceinline__ void store_bytes(int8_t *dense8, long long e0, const float (&f)[V]) {
    unsigned pk[V / 4];
    pack_bytes<V>(f, pk);
    if (V == 4) *reinterpret_cast<unsigned *>(dense8 + e0) = pk[0];
    else *reinterpret_cast<uint2 *>(dense8 + e0) = make_uint2(pk[0], pk[V / 4 - 1]);
}

// Three ways to fill a tile:
//   kFlat: planes smaller than a tile's 64 positions (C % 8 == 0): the tile's 64 channels of one image are one contiguous
//          run of delta_z, read as whole vectors whatever the plane size;
//   kPair: plane size % V == 0: a thread takes the same V positions of two neighbouring channels and writes the two codes
//          of a position as one word;
//   kOdd:  any other plane: a channel's row of the tile is covered by the aligned vectors that touch it (one more than a
//          row holds), and what lies outside the row is dropped.
// The output's rows are padded to a multiple of eight channels (the padding is not written: the copy engine never reads
// it). The first tile's loads and dithers, and every next tile's loads, are under way before they are needed (see above).
enum { kFlat, kPair, kOdd };

template <typename T, int V, int PATH, bool STACK, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_nhwc_kernel(const T *__restrict__ x, int B, int C, int HW, unsigned long long seed, const StepSource step,
                     unsigned short *__restrict__ out, int8_t *__restrict__ dense8, DeviceState *__restrict__ st, int count,
                     unsigned short *__restrict__ out_stack, int plane_w, const unsigned char *__restrict__ mask) {
    __shared__ __align__(16) unsigned char tile[2][kTileBytes];
    constexpr int VPR = kTP / V;                                   // kPair: vectors per channel row of the tile
    constexpr int NI = kTC * kTP / V / kThreads;                   // vectors per thread and tile (kFlat: at most)
    const unsigned ct = (C + kTC - 1) / kTC, pt = (HW + kTP - 1) / kTP, per_img = ct * pt, ntiles = B * per_img;
    const int pitch = (C + 7) & ~7;

    uint4 raw[NI];
    unsigned msk[MASKED ? NI : 1];
    unsigned long long u[NI][V / 2];
    struct Tile { int b, c0, p0; };
    auto tile_of = [&](unsigned t) {
        Tile r;
        r.b = t / per_img;
        const unsigned rem = t - r.b * per_img;
        r.c0 = (rem / pt) * kTC;
        r.p0 = (rem - rem / pt * pt) * kTP;
        return r;
    };
    // vector i of this thread: its first element, and whether it exists
    auto vec_of = [&](const Tile &tl, int i, long long &e0) {
        if (PATH == kFlat) {
            const int v = threadIdx.x + kThreads * i, nch = C - tl.c0 < kTC ? C - tl.c0 : kTC;
            e0 = (static_cast<long long>(tl.b) * C + tl.c0) * HW + v * V;
            return v * V < nch * HW;
        }
        const int it = threadIdx.x + kThreads * (i >> 1), c = 2 * (it / VPR) + (i & 1), pv = (it % VPR) * V;
        e0 = (static_cast<long long>(tl.b) * C + tl.c0 + c) * HW + tl.p0 + pv;
        return tl.c0 + c < C && tl.p0 + pv < HW;
    };
    auto load = [&](const Tile &tl) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            long long e0;
            const bool in = vec_of(tl, i, e0);
            raw[i] = in ? load_raw<T, V>(x + e0) : make_uint4(0u, 0u, 0u, 0u);
            if (MASKED) msk[i] = in ? mask_word(mask, e0) : 0u;
        }
    };
    auto draw = [&](const Tile &tl) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            long long e0;
            vec_of(tl, i, e0);
            dithers_of<V>(e0, seed, u[i]);
        }
    };
    unsigned t = blockIdx.x;
    Tile cur = tile_of(t);
    if (PATH != kOdd) {
        load(cur);
        draw(cur);
    }
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(step, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned nnz = 0, sat = 0, nz2 = 0;
    int buf = 0;
    for (; t < ntiles; buf ^= 1) {
        unsigned char *tl = tile[buf];
        const int b = cur.b, c0 = cur.c0, p0 = cur.p0;
        const unsigned next = t + gridDim.x;
        const Tile nxt = tile_of(next < ntiles ? next : t);
        if (PATH != kOdd) {
            float f[NI][V];
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                float v[V];
                values_of(x, raw[i], v);
                if (MASKED) apply_mask(msk[i], v);
                decide<V>(v, u[i], inv, f[i], sat);
            }
            load(nxt);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                long long e0;
                if (vec_of(cur, i, e0)) {
                    unsigned h[V / 2];
                    pack_bf16<V>(f[i], h);
                    count_pairs<V>(h, nz2);
                    if (dense8 != nullptr) store_bytes<V>(dense8, e0, f[i]);
                    if (PATH == kFlat) {
                        const int v = threadIdx.x + kThreads * i;
                        int c = (v * V) / HW, pp = v * V - c * HW;
#pragma unroll
                        for (int j = 0; j < V; ++j) {
                            *reinterpret_cast<unsigned short *>(tl + tile_off(pp, c)) = static_cast<unsigned short>(h[j >> 1] >> (16 * (j & 1)));
                            if (++pp == HW) { pp = 0; ++c; }
                        }
                    }
                }
            }
            if (PATH == kPair) {
                // (a vector that does not exist was decided as zeros: code 0, never stored beyond the tile)
#pragma unroll
                for (int i = 0; i < NI / 2; ++i) {
                    const int it = threadIdx.x + kThreads * i, c = 2 * (it / VPR), pv = (it % VPR) * V;
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        *reinterpret_cast<unsigned *>(tl + tile_off(pv + j, c)) =
                            __byte_perm(__float_as_uint(f[2 * i][j]), __float_as_uint(f[2 * i + 1][j]), 0x7632);
                }
            }
            if (next < ntiles) draw(nxt);
        } else {
            constexpr int VO = kTP / V + 1;                        // aligned vectors that may touch a row of the tile
            const int len = HW - p0 < kTP ? HW - p0 : kTP, nch = C - c0 < kTC ? C - c0 : kTC;
            const long long total = static_cast<long long>(B) * C * HW;
            for (int it = threadIdx.x; it < nch * VO; it += kThreads) {
                const int c = it / VO;
                const long long row0 = (static_cast<long long>(b) * C + c0 + c) * HW + p0;
                const long long e0 = (row0 & ~static_cast<long long>(V - 1)) + (it - c * VO) * V;
                const int pp = static_cast<int>(e0 - row0);        // position of the vector's first element in the row
                if (pp >= len) continue;
                float v[V], f[V];
                if (e0 + V <= total) {
                    values_of(x, load_raw<T, V>(x + e0), v);
                    if (MASKED) apply_mask(mask_word(mask, e0), v);
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j)
                        v[j] = e0 + j < total && (!MASKED || __ldg(mask + e0 + j)) ? Vec<T>::one(x + e0 + j) : 0.f;
                }
                // what lies outside the row belongs to other rows: it is not counted here, clipped or not
#pragma unroll
                for (int j = 0; j < V; ++j) v[j] = pp + j >= 0 && pp + j < len ? v[j] : 0.f;
                dithers_of<V>(e0, seed, u[0]);
                decide<V>(v, u[0], inv, f, sat);
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (pp + j >= 0 && pp + j < len) {
                        nnz += f[j] != 0.f;
                        *reinterpret_cast<unsigned short *>(tl + tile_off(pp + j, c)) = static_cast<unsigned short>(__float_as_uint(f[j]) >> 16);
                        if (dense8 != nullptr) dense8[e0 + j] = static_cast<int8_t>(static_cast<int>(f[j]));
                    }
            }
        }
        __syncthreads();
        // rows of 64 channels (128 bytes) of one position each; eight lanes per row
#pragma unroll
        for (int i = 0; i < (kTP * 8) / kThreads; ++i) {
            const int v = threadIdx.x + kThreads * i;
            const int pp = v >> 3, ch = v & 7;
            if (p0 + pp < HW && c0 + ch * 8 < C)
                *reinterpret_cast<uint4 *>(out + (static_cast<long long>(b) * HW + p0 + pp) * pitch + c0 + ch * 8) =
                    *reinterpret_cast<const uint4 *>(tl + tile_off(pp, ch * 8));
            // Second copy for the weight-gradient kernel of tiny planes: the images one below the other as tall
            // images, a row of zeros after every image (what a tap that leaves an image must read).
            if (STACK && pp < HW + plane_w && c0 + ch * 8 < C) {
                const uint4 val = pp < HW ? *reinterpret_cast<const uint4 *>(tl + tile_off(pp, ch * 8)) : make_uint4(0u, 0u, 0u, 0u);
                const long long row = static_cast<long long>(b) * (HW + plane_w) + pp;   // any number of images per tall image
                *reinterpret_cast<uint4 *>(out_stack + row * C + c0 + ch * 8) = val;
            }
        }
        // the other buffer is written next; this one again only after the next barrier
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
        t = next;
        cur = nxt;
    }
    nnz += pairs_total(nz2);
    if (count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}

template <typename T, int V, int PATH>
cudaError_t run_nhwc(dbp_ctx *ctx, const void *delta, int B, int C, int HW, unsigned long long seed, const StepSource &step,
                     void *out, int8_t *dense8, bool count, void *out_stack, int plane_w, const uint8_t *mask) {
    const long long ntiles = static_cast<long long>(B) * ((C + kTC - 1) / kTC) * ((HW + kTP - 1) / kTP);
    const long long cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM, blocks = ntiles < cap ? ntiles : cap;
    auto go = [&](auto kern) {
        return launch_chained(kern, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream,
                              static_cast<const T *>(delta), B, C, HW, seed, step, static_cast<unsigned short *>(out), dense8,
                              ctx->state, count ? 1 : 0, static_cast<unsigned short *>(out_stack), plane_w,
                              static_cast<const unsigned char *>(mask));
    };
    if constexpr (sizeof(T) == 4) {
        if (mask != nullptr) {
            if constexpr (PATH == kFlat) { if (out_stack) return go(quantize_nhwc_kernel<T, V, PATH, true, true>); }
            return go(quantize_nhwc_kernel<T, V, PATH, false, true>);
        }
    }
    if constexpr (PATH == kFlat) { if (out_stack) return go(quantize_nhwc_kernel<T, V, PATH, true, false>); }
    return go(quantize_nhwc_kernel<T, V, PATH, false, false>);
}

// ---------------------------------------------------------------- bf16 planes of odd sizes
// Planes whose size is no multiple of 4 (7 x 7, 9 x 9, ...) written at a pitch that is a multiple of 8: the codes
// of eight consecutive elements then belong to unaligned places of one or two planes. A block takes a run of
// whole planes (a multiple of eight of them, so that the run starts on a 16-byte boundary and on an even
// element), quantizes it with whole-vector loads as everywhere, places the codes in shared memory at their pitch,
// and the run leaves as one contiguous copy (the padding of a plane is never read by anybody).
constexpr int kOddMaxSmem = 12 * 1024;            // bytes of the staged run (planes x pitch bf16)

template <typename T, bool MASKED>
__global__ void __launch_bounds__(kThreads)
quantize_planes_odd_kernel(const T *__restrict__ x, long long nplanes, int hw, int pitch, int planes_per_run,
                           unsigned long long seed, const StepSource step, unsigned short *__restrict__ out,
                           int8_t *__restrict__ dense8, DeviceState *__restrict__ st, int count,
                           const unsigned char *__restrict__ mask) {
    constexpr int V = Vec<T>::V;
    constexpr int NP = 2;                                           // vectors of the first run loaded and drawn ahead
    __shared__ __align__(16) unsigned short run_s[kOddMaxSmem / 2];
    const long long nruns = (nplanes + planes_per_run - 1) / planes_per_run;
    uint4 raw[NP];
    unsigned long long u[NP][V / 2];
    {
        const long long e_base = blockIdx.x * static_cast<long long>(planes_per_run) * hw, n = nplanes * hw;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const long long e0 = e_base + (threadIdx.x + kThreads * i) * V;
            raw[i] = e0 < n ? Vec<T>::raw(x + e0) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < NP; ++i) dithers_of<V>(e_base + (threadIdx.x + kThreads * i) * V, seed, u[i]);
    }
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(step, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned sat = 0, nz2 = 0, nnz = 0;
    for (long long r = blockIdx.x; r < nruns; r += gridDim.x) {
        const long long pl0 = r * planes_per_run;
        const int np = static_cast<int>(nplanes - pl0 < planes_per_run ? nplanes - pl0 : planes_per_run);   // a multiple of 8
        const long long e_base = pl0 * hw;
        const int nvec = np * hw / V;
        auto place = [&](int v, const uint4 &q, const unsigned long long (&d)[V / 2]) {
            float a[V], f[V];
            unsigned h[V / 2];
            Vec<T>::values(q, a);
            if (MASKED) apply_mask(mask_word(mask, e_base + static_cast<long long>(v) * V), a);
            decide<V>(a, d, inv, f, sat);
            pack_bf16<V>(f, h);
            count_pairs<V>(h, nz2);
            if (dense8 != nullptr) store_bytes<V>(dense8, e_base + static_cast<long long>(v) * V, f);
            int pl = (v * V) / hw, pp = v * V - pl * hw;
#pragma unroll
            for (int j = 0; j < V; ++j) {
                run_s[pl * pitch + pp] = static_cast<unsigned short>(h[j >> 1] >> (16 * (j & 1)));
                if (++pp == hw) { pp = 0; ++pl; }
            }
        };
        int v = threadIdx.x;
        if (r == blockIdx.x) {
#pragma unroll
            for (int i = 0; i < NP; ++i, v += kThreads)
                if (v < nvec) place(v, raw[i], u[i]);
        }
        for (; v < nvec; v += kThreads) {
            const long long e0 = e_base + static_cast<long long>(v) * V;
            const uint4 q = Vec<T>::raw(x + e0);
            unsigned long long d[V / 2];
            dithers_of<V>(e0, seed, d);
            place(v, q, d);
        }
        __syncthreads();
        const int n16 = np * pitch / 8;
        uint4 *dst = reinterpret_cast<uint4 *>(out + pl0 * pitch);
        for (int i = threadIdx.x; i < n16; i += kThreads) dst[i] = reinterpret_cast<const uint4 *>(run_s)[i];
        __syncthreads();
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
    }
    nnz += pairs_total(nz2);
    if (count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}

}  // namespace

int launch_quantize_dense(dbp_ctx *ctx, const void *delta, int dtype, long long numel,
                          unsigned long long seed, const StepSource &step, int8_t *dense,
                          void *planes_bf16, long long hw, long long pitch, bool count, const uint8_t *mask) {
    if (mask != nullptr && dtype != DBP_F32) return DBP_EUNSUPPORTED;
    const unsigned char *m = static_cast<const unsigned char *>(mask);
    unsigned short *planes = static_cast<unsigned short *>(planes_bf16);
    const int v = dtype == DBP_F32 ? 4 : 8;
    const float *xf = static_cast<const float *>(delta);
    const __nv_bfloat16 *xb = static_cast<const __nv_bfloat16 *>(delta);
    // odd plane sizes at a padded pitch: whole runs of planes through shared memory
    if (planes != nullptr && hw > 0 && pitch != hw && (hw & 3) != 0 && numel % hw == 0 && (numel / hw) % 8 == 0 &&
        8 * pitch * 2 <= kOddMaxSmem && hw < (1 << 20)) {
        const long long nplanes = numel / hw;
        int per_run = static_cast<int>(kOddMaxSmem / 2 / pitch / 8 * 8);          // planes per run: a multiple of 8
        const long long want = (4096 + 8 * hw - 1) / (8 * hw) * 8;               // about 4096 elements a run
        if (per_run > want) per_run = static_cast<int>(want);
        const long long nruns = (nplanes + per_run - 1) / per_run, cap = static_cast<long long>(ctx->sm_count) * 8;
        auto go = [&](auto kern, auto x) {
            return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(nruns < cap ? nruns : cap)), dim3(kThreads), 0, ctx->stream, x,
                                          nplanes, static_cast<int>(hw), static_cast<int>(pitch), per_run, seed, step, planes, dense,
                                          ctx->state, count ? 1 : 0, m));
        };
        return dtype != DBP_F32 ? go(quantize_planes_odd_kernel<__nv_bfloat16, false>, xb)
               : m              ? go(quantize_planes_odd_kernel<float, true>, xf)
                                : go(quantize_planes_odd_kernel<float, false>, xf);
    }
    long long blocks = (numel / v + 2 * kThreads - 1) / (2 * kThreads);
    if (blocks < 1) blocks = 1;
    const long long cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM;
    if (blocks > cap) blocks = cap;
    const CodeSinks out{dense, planes, hw > 0 ? hw : 1, pitch > 0 ? pitch : 1, count ? 1 : 0};
    auto go = [&](auto kern, auto x) {
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream, x, numel, seed, step, out,
                                      ctx->state, m));
    };
    return dtype != DBP_F32 ? go(quantize_dense_kernel<__nv_bfloat16, false>, xb)
           : m              ? go(quantize_dense_kernel<float, true>, xf)
                            : go(quantize_dense_kernel<float, false>, xf);
}

// delta_z [B][C][HW] -> bf16 codes [B][HW][C rounded up to a multiple of 8] and, when dense8 is not null, int8 codes
// in delta_z's order
int launch_quantize_nhwc(dbp_ctx *ctx, const void *delta, int dtype, long long B, long long C, long long HW,
                         unsigned long long seed, const StepSource &step, void *codes_nhwc, int8_t *dense8, bool count,
                         void *codes_stack, int plane_w, const uint8_t *mask) {
    if (B * C * HW >= (1ll << 40) || HW >= (1ll << 30)) return DBP_EUNSUPPORTED;
    if (B * ((C + kTC - 1) / kTC) * ((HW + kTP - 1) / kTP) >= (1ll << 31)) return DBP_EUNSUPPORTED;
    if (mask != nullptr && dtype != DBP_F32) return DBP_EUNSUPPORTED;
    // the stacked copy is written by the path for planes smaller than a tile; the rows of image b start at
    // b (HW + W) however many images make up a tall image: the stacking only adds the zero rows
    if (codes_stack != nullptr && (HW >= kTP || C % 8 != 0 || plane_w <= 0 || HW + plane_w > kTP)) return DBP_EINVAL;
    const int b = static_cast<int>(B), c = static_cast<int>(C), hw = static_cast<int>(HW);
    const bool flat = HW < kTP && C % 8 == 0;
    auto run = [&](auto kern) { return kern(ctx, delta, b, c, hw, seed, step, codes_nhwc, dense8, count, codes_stack, plane_w, mask); };
    if (dtype == DBP_F32)
        return cuda_ok(flat          ? run(run_nhwc<float, 4, kFlat>)
                       : hw % 4 == 0 ? run(run_nhwc<float, 4, kPair>)
                                     : run(run_nhwc<float, 4, kOdd>));
    return cuda_ok(flat          ? run(run_nhwc<__nv_bfloat16, 8, kFlat>)
                   : hw % 8 == 0 ? run(run_nhwc<__nv_bfloat16, 8, kPair>)
                   : hw % 4 == 0 ? run(run_nhwc<__nv_bfloat16, 4, kPair>)
                                 : run(run_nhwc<__nv_bfloat16, 8, kOdd>));
}

}  // namespace dbp
