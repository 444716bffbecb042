// NSD quantization for the product kernels (Section 3.1, Eq. (nsd)): the same codes as quantize_kernel, written only as
// the dense arrays the dX / dW kernels read, without the bitmap / offsets / packed-values structure. Used when the caller
// did not ask for the sparse structure, so the pass costs one read of delta_z and one write of the codes.
//
// What bounds the kernels are instructions: 16 per element are the decision, 11.5 of them the SplitMix64 draw (nsd_common.cuh), so
// that the rest is kept small: pairs per instruction, addresses and counters by constants, one test for care per tile. 12.8 M
// bf16 elements: 13.8 us, by vectors with their own bounds and branches 19.1 (32 instructions an element). A thread's first vectors of
// delta_z and their dithers need
// nothing of the statistics kernel that runs before: they are loaded and drawn before the wait for it. That is safe
// because the statistics kernel lets this one start only once all of its own blocks have seen the kernels before it
// complete. In the loop the next vectors are loaded before the current ones are stored.
#include "nsd_common.cuh"

#include <type_traits>

namespace dbp {

namespace {

using namespace nsd;

constexpr int kThreads = 256;
constexpr int kBlocksPerSM = 3;                   // resident blocks the dense quantizer is compiled for

// Where the codes of the flat quantizer go:
//   kBytes: one byte per element, same order as delta_z;
//   kSame:  bf16, same order;
//   kPad4:  bf16 as [plane][hw + 4], planes of an odd multiple of four elements (so every plane starts on a 16-byte boundary).
// (Planes of other sizes: quantize_rows_kernel.)
enum { kBytes, kSame, kPad4 };
struct CodeSinks {
    int8_t *dense8;
    unsigned short *planes16;
    long long hw, pitch;
    // kPad4: from one of a thread's vectors to the next, and from its last one of a tile to the first of its next tile: whole
    // planes and a rest, as the rest (elements) and the distance in the output without a plane's end between them
    int rest1, rest2;
    long long dist1, dist2;
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

__device__ __forceinline__ void store_code(const CodeSinks &o, long long e, unsigned byte) {
    if (o.dense8 != nullptr) o.dense8[e] = static_cast<int8_t>(byte);
    if (o.planes16 != nullptr) {
        const long long plane = e / o.hw;
        const float f = static_cast<float>(static_cast<int>(static_cast<signed char>(byte)));
        o.planes16[plane * o.pitch + (e - plane * o.hw)] = static_cast<unsigned short>(__float_as_uint(f) >> 16);
    }
}
template <int V>
__device__ __forceinline__ void store_vec(unsigned short *dst, const unsigned (&h)[V / 2]) {
    if (V == 4) *reinterpret_cast<uint2 *>(dst) = make_uint2(h[0], h[1]);
    else *reinterpret_cast<uint4 *>(dst) = make_uint4(h[0], h[1], h[V / 2 - 2], h[V / 2 - 1]);
}

// mask (fp32 tensors only): x is delta_a and the gradient is delta_a where mask != 0, else 0. The four mask bytes of a
// vector as one word.
__device__ __forceinline__ unsigned mask_word(const unsigned char *mask, long long e) { return __ldg(reinterpret_cast<const unsigned *>(mask + e)); }
__device__ __forceinline__ void apply_mask(unsigned m, float (&v)[4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (m >> (8 * j)) & 0xffu ? v[j] : 0.f;
}
__device__ __forceinline__ void apply_mask(unsigned, float (&)[8]) {}                 // bf16 tensors take no mask

// A block takes tiles of 16 elements per thread: a thread's vectors lie 256 vectors apart, so that within a tile every address
// and every counter of the dither is the first one's plus a constant, and from tile to tile all of them advance by constants.
constexpr int kPerThread = 16;

// A gradient that the statistics kernel writes (LATE) is read behind the wait for it, by loads that are no read-only ones and
// that the compiler leaves in their places.
__device__ __forceinline__ uint4 load_written(const void *p) {
    uint4 v;
    asm volatile("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
    return v;
}

template <typename T, bool MASKED, int SINK, bool LATE = false>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_dense_kernel(const T *__restrict__ x, long long n, unsigned long long seed, const StepSource step,
                      const __grid_constant__ CodeSinks out, DeviceState *__restrict__ st, const unsigned char *__restrict__ mask) {
    constexpr int V = Vec<T>::V, NV = kPerThread / V, kTile = kThreads * kPerThread;
    constexpr int kBetween = kThreads * V;                             // elements between two vectors of a thread
    constexpr unsigned long long kBetweenZ = kBetween / 2 * kGamma;
    const long long nvec = n / V, whole = nvec / (kTile / V);          // whole tiles; the next one holds what is left
    const int ragged = static_cast<int>(nvec - whole * (kTile / V));   // vectors
    const long long ntile = whole + (ragged > 0);
    const long long stride_e = static_cast<long long>(gridDim.x) * kTile;
    const unsigned long long stride_z = static_cast<unsigned long long>(stride_e / 2) * kGamma;
    long long t = blockIdx.x;
    long long e0 = t * kTile + threadIdx.x * V;                        // the thread's first element of the tile
    unsigned long long z = counter_of(e0, seed);
    uint4 raw[NV];
    unsigned msk[MASKED ? NV : 1];
    unsigned long long u[NV][V / 2];
    auto vec = [&](const T *p) { return LATE ? load_written(p) : Vec<T>::raw(p); };
    auto there = [&](int k) { return static_cast<int>(threadIdx.x) + k * kThreads < ragged; };      // in the tile after the whole ones
    auto load = [&](long long tile, long long e) {
        if (tile < whole) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                raw[k] = vec(x + e + k * kBetween);
                if (MASKED) msk[k] = mask_word(mask, e + k * kBetween);
            }
        } else if (tile == whole) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                raw[k] = there(k) ? vec(x + e + k * kBetween) : make_uint4(0u, 0u, 0u, 0u);
                if (MASKED) msk[k] = there(k) ? mask_word(mask, e + k * kBetween) : 0u;
            }
        }
    };
    auto draw = [&](unsigned long long zz) {
#pragma unroll
        for (int k = 0; k < NV; ++k) dithers_at<V>(zz + k * kBetweenZ, u[k]);
    };
    if (!LATE) load(t, e0);
    draw(z);
    keep_here(u);
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    if (LATE) load(t, e0);
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: x * 0 + u < 1, every code 0 (NaN too)
    unsigned sat = 0, nz2 = 0, nnz = 0;
    int pp = 0;                                                        // kPad4: place in the plane
    unsigned short *po = out.planes16;                                 // and in the output
    if (SINK == kPad4 && t < ntile) {
        long long plane, r;
        split_index(e0, out.hw, plane, r);
        pp = static_cast<int>(r);
        po += plane * (out.hw + 4) + r;
    }
    // vector k of the tile at e goes out; pp and po walk from one of the thread's vectors to its next
    auto store = [&](long long e, int k, const unsigned (&h)[V / 2], const unsigned (&m)[V]) {
        if (SINK == kBytes) {
            unsigned pk[V / 4];
            low_bytes<V>(m, pk);
            int8_t *dst = out.dense8 + e + k * kBetween;
            if (V == 4) *reinterpret_cast<unsigned *>(dst) = pk[0];
            else *reinterpret_cast<uint2 *>(dst) = make_uint2(pk[0], pk[V / 4 - 1]);
        } else if (SINK == kSame) {
            store_vec<V>(out.planes16 + e + k * kBetween, h);
        } else {
            // each group of four codes lies in one plane and starts on an 8-byte boundary there
            *reinterpret_cast<uint2 *>(po) = make_uint2(h[0], h[1]);
            if (V == 8) {
                if (pp + 4 < static_cast<int>(out.hw)) *reinterpret_cast<uint2 *>(po + 4) = make_uint2(h[V / 2 - 2], h[V / 2 - 1]);
                else *reinterpret_cast<uint2 *>(po + 8) = make_uint2(h[V / 2 - 2], h[V / 2 - 1]);
            }
        }
    };
    auto walk = [&](int k) {
        if (SINK != kPad4) return;
        pp += k + 1 < NV ? out.rest1 : out.rest2;
        po += k + 1 < NV ? out.dist1 : out.dist2;
        if (pp >= static_cast<int>(out.hw)) { pp -= static_cast<int>(out.hw); po += 4; }
    };
    for (; t < ntile; t += gridDim.x) {
        unsigned h[NV][V / 2], m[NV][V], top = 0u;
        const unsigned before = nz2;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            float v[V];
            Vec<T>::values(raw[k], v);
            if (MASKED) apply_mask(msk[k], v);
            quick_codes<V>(v, u[k], inv, h[k], m[k], top);
            count_pairs<V>(h[k], nz2);                                 // (a vector that does not exist is zeros: code 0)
        }
        const long long e = e0;
        e0 += stride_e;
        load(t + gridDim.x, e0);
        if (needs_care(top)) {                                         // rare: clip, count, NaN
            nz2 = before;
#pragma unroll 1
            for (int k = 0; k < NV; ++k) {
                if (t < whole || there(k)) {
                    float v[V];
                    unsigned long long d[V / 2];
                    unsigned hc[V / 2], mc[V];
                    Vec<T>::values(vec(x + e + k * kBetween), v);
                    if (MASKED) apply_mask(mask_word(mask, e + k * kBetween), v);
                    dithers_at<V>(z + k * kBetweenZ, d);
                    careful_codes<V>(v, d, inv, hc, mc, sat);
                    count_pairs<V>(hc, nz2);
                    store(e, k, hc, mc);
                }
                walk(k);
            }
        } else if (t < whole) {
#pragma unroll
            for (int k = 0; k < NV; ++k) { store(e, k, h[k], m[k]); walk(k); }
        } else {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                if (there(k)) store(e, k, h[k], m[k]);
                walk(k);
            }
        }
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
        z += stride_z;
        if (t + gridDim.x < ntile) draw(z);
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
// 64 channels x up to 64 positions through shared memory: rows of the input are read along the
// positions, rows of the output are written along the channels. The dither of an element is
// still keyed on its index in delta_z's own order. The output's rows are padded to a multiple of eight channels (the
// padding is not written: the copy engine never reads it).
//
// Planes of a multiple of V elements. A tile is P positions of one image, or G whole images of small planes (P = HW); a thread
// takes the same V positions of two neighbouring channels, NI times, and writes the two codes of a position as one word.
// Where these lie in a tile, in the input, in shared memory and in the dither's sequence is the same for every tile and made
// once; what changes from tile to tile is the same for all threads. The first tile's loads and dithers, and every next tile's
// loads, are under way before they are needed (see above).
constexpr int kTC = 64, kTP = 64;                 // channels, most positions of a tile
constexpr int kTileBytes = kTP * kTC * 2;

// shared-memory byte offset of (position p, channel c) inside a tile: 128-byte rows, the 16-byte pieces of a row permuted by
// the number of the row's group of V (the eight groups and four channel pairs of a warp's words lie in different banks)
template <int V>
__device__ __forceinline__ unsigned tile_off(int p, int c) {
    return static_cast<unsigned>(p) * 128u + (((static_cast<unsigned>(c) >> 3) ^ ((static_cast<unsigned>(p) / V) & 7u)) << 4) +
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

struct NhwcP {
    int B, C, HW;
    int P, G;                     // positions of an image, images of a tile
    int pt, ct, ntiles;           // tiles along the positions, along the channels, in all (positions first, images last)
    // From one of a block's tiles to its next: tiles along the positions, the channels and the images, and how much further
    // everything is then that grows from tile to tile: the place in delta_z (elements), in the output, in the stacked copy, and
    // the dither's counter. wrap_p: after that where the positions pass their end, wrap_c where the channels do.
    int step_p, step_c, step_b;
    struct Far { long long in, out, tall; unsigned long long z; } far, wrap_p, wrap_c;
    int plane_w;                  // stacked copy: rows of zeros after every image
    int count;
};

template <typename T, int V, bool STACK, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_nhwc_kernel(const T *__restrict__ x, const NhwcP p, unsigned long long seed, const StepSource step,
                     unsigned short *__restrict__ out, unsigned short *__restrict__ out_stack, DeviceState *__restrict__ st,
                     const unsigned char *__restrict__ mask) {
    __shared__ __align__(16) unsigned char tile[2][kTileBytes];
    constexpr int NI = kTC * kTP / (2 * V) / kThreads;             // pairs of vectors per thread and tile (at most)
    const int C = p.C, HW = p.HW, pitch = (C + 7) & ~7;
    const unsigned long long row_z = static_cast<unsigned long long>(HW / 2) * kGamma;

    // this thread's pairs of vectors in any tile: four channel pairs run fastest, then the positions, eights of channels, images
    int in_off[NI], row[NI], ch[NI];                               // first element; first row of the tile; first channel
#pragma unroll
    for (int i = 0; i < NI; ++i) {
        const int s = threadIdx.x + kThreads * i, vpr = p.P / V, q = s >> 2, r = q / vpr, pv = (q - r * vpr) * V, g = r >> 3;
        ch[i] = 8 * (r & 7) + 2 * (s & 3);
        row[i] = g < p.G ? g * p.P + pv : kTP;                     // kTP: in no tile
        in_off[i] = (g * C + ch[i]) * HW + pv;
    }
    auto off_z = [&](int i) { return static_cast<unsigned long long>(static_cast<unsigned>(in_off[i]) >> 1) * kGamma; };
    // the tile: numbers along the positions, the channels and the images; places of its first element; rows and channels it has
    struct Tile { int p, c, b; long long e; unsigned long long z; unsigned short *out, *tall; int rows, cleft; };
    auto measure = [&](Tile &t) {
        const int n = p.G == 1 ? HW - t.p * p.P : (p.B - t.b * p.G) * HW;
        t.rows = n < p.G * p.P ? n : p.G * p.P;
        t.cleft = C - t.c * kTC;
    };
    auto go_in = [&](Tile &t, const NhwcP::Far &f) { t.e += f.in; t.z += f.z; };
    auto go_out = [&](Tile &t, const NhwcP::Far &f) { t.out += f.out; if (STACK) t.tall += f.tall; };
    uint4 raw[NI][2];
    unsigned msk[MASKED ? NI : 1][2];
    unsigned long long u[NI][2][V / 2];
    auto load = [&](const Tile &t) {
        if (t.cleft >= kTC && t.rows == kTP) {                     // a whole tile
#pragma unroll
            for (int i = 0; i < NI; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    raw[i][h] = load_raw<T, V>(x + t.e + in_off[i] + h * HW);
                    if (MASKED) msk[i][h] = mask_word(mask, t.e + in_off[i] + h * HW);
                }
        } else {
#pragma unroll
            for (int i = 0; i < NI; ++i)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const bool in = row[i] < t.rows && ch[i] + h < t.cleft;
                    raw[i][h] = in ? load_raw<T, V>(x + t.e + in_off[i] + h * HW) : make_uint4(0u, 0u, 0u, 0u);
                    if (MASKED) msk[i][h] = in ? mask_word(mask, t.e + in_off[i] + h * HW) : 0u;
                }
        }
    };
    auto draw = [&](const Tile &t) {
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (row[i] >= t.rows) continue;
            dithers_at<V>(t.z + off_z(i), u[i][0]);
            dithers_at<V>(t.z + off_z(i) + row_z, u[i][1]);
        }
    };
    unsigned t = blockIdx.x;
    const unsigned ntiles = p.ntiles;
    // rows on the way out: eight lanes to a row of 64 channels, thread 8 r + k at row r and r + 32
    const int orow = threadIdx.x >> 3, och = (threadIdx.x & 7) * 8;
    auto tile_at = [&](unsigned n) {
        Tile r;
        r.b = n / (p.pt * p.ct);
        r.c = (n - r.b * p.pt * p.ct) / p.pt;
        r.p = n - (r.b * p.ct + r.c) * p.pt;
        const long long b0 = static_cast<long long>(r.b) * p.G;
        r.e = (b0 * C + r.c * kTC) * HW + r.p * p.P;
        r.z = counter_of(r.e, seed);
        r.out = out + (b0 * HW + r.p * p.P + orow) * pitch + r.c * kTC + och;
        r.tall = out_stack + b0 * (HW + p.plane_w) * C + r.c * kTC + och;
        measure(r);
        return r;
    };
    Tile cur = tile_at(t);
    load(cur);
    draw(cur);
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned nnz = 0, sat = 0, nz2 = 0;
    for (int buf = 0; t < ntiles; buf ^= 1) {
        unsigned char *tl = tile[buf];
        const int rows = cur.rows, cleft = cur.cleft;
        t += gridDim.x;
        cur.p += p.step_p;
        cur.c += p.step_c;
        cur.b += p.step_b;
        const bool past_p = cur.p >= p.pt;
        go_in(cur, p.far);
        if (past_p) { cur.p -= p.pt; ++cur.c; go_in(cur, p.wrap_p); }
        const bool past_c = cur.c >= p.ct;
        if (past_c) { cur.c -= p.ct; ++cur.b; go_in(cur, p.wrap_c); }
        measure(cur);
        unsigned w[NI][V], top = 0u;
        const unsigned before = nz2;
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (row[i] >= rows) continue;
            float a[V], b[V];
            values_of(x, raw[i][0], a);
            values_of(x, raw[i][1], b);
            if (MASKED) { apply_mask(msk[i][0], a); apply_mask(msk[i][1], b); }
            quick_codes2<V>(a, b, u[i][0], u[i][1], inv, w[i], top);
            count_pairs<2 * V>(w[i], nz2);
        }
        if (t < ntiles) load(cur);
        if (needs_care(top)) {                                     // rare: clip, count, NaN
            nz2 = before;
            const Tile now = tile_at(t - gridDim.x);
#pragma unroll
            for (int i = 0; i < NI; ++i) {
                if (row[i] >= rows) continue;
                unsigned m[2][V];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    float v[V];
                    unsigned long long d[V / 2];
                    unsigned hc[V / 2];
                    const bool in = ch[i] + h < cleft;
                    values_of(x, in ? load_raw<T, V>(x + now.e + in_off[i] + h * HW) : make_uint4(0u, 0u, 0u, 0u), v);
                    if (MASKED) apply_mask(in ? mask_word(mask, now.e + in_off[i] + h * HW) : 0u, v);
                    dithers_at<V>(now.z + off_z(i) + h * row_z, d);
                    careful_codes<V>(v, d, inv, hc, m[h], sat);
                }
#pragma unroll
                for (int j = 0; j < V; ++j)
                    w[i][j] = __byte_perm(__float_as_uint(__uint_as_float(m[0][j]) - kMagic),
                                          __float_as_uint(__uint_as_float(m[1][j]) - kMagic), 0x7632);
                count_pairs<2 * V>(w[i], nz2);
            }
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) {
            if (row[i] >= rows) continue;
            unsigned char *dst = tl + tile_off<V>(row[i], ch[i]);
#pragma unroll
            for (int j = 0; j < V; ++j) *reinterpret_cast<unsigned *>(dst + j * 128) = w[i][j];
        }
        if (t < ntiles) draw(cur);
        __syncthreads();
        if (och < cleft) {
#pragma unroll
            for (int i = 0; i < kTP / 32; ++i)
                if (orow + 32 * i < rows)
                    *reinterpret_cast<uint4 *>(cur.out + static_cast<long long>(32 * i) * pitch) =
                        *reinterpret_cast<const uint4 *>(tl + tile_off<V>(orow + 32 * i, och));
            // Second copy for the weight-gradient kernel of tiny planes: the images one below the other as tall images, a row of
            // zeros after every image (what a tap that leaves an image must read). Any number of images per tall image.
            if (STACK) {
#pragma unroll
                for (int i = 0; i < kTP / 32; ++i) {
                    const int r = orow + 32 * i, g = r / HW;
                    if (r < rows)
                        *reinterpret_cast<uint4 *>(cur.tall + static_cast<long long>(r + g * p.plane_w) * C) =
                            *reinterpret_cast<const uint4 *>(tl + tile_off<V>(r, och));
                }
                const int images = rows / HW;
                for (int r = orow; r < images * p.plane_w; r += 32) {
                    const int g = r / p.plane_w;
                    *reinterpret_cast<uint4 *>(cur.tall + static_cast<long long>((g + 1) * HW + r) * C) = make_uint4(0u, 0u, 0u, 0u);
                }
            }
        }
        go_out(cur, p.far);
        if (past_p) go_out(cur, p.wrap_p);
        if (past_c) go_out(cur, p.wrap_c);
        // the other buffer is written next; this one again only after the next barrier
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
    }
    nnz += pairs_total(nz2);
    if (p.count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}

template <typename T, int V>
cudaError_t run_nhwc(dbp_ctx *ctx, const void *delta, int B, int C, int HW, unsigned long long seed, const StepSource &step,
                     void *out, bool count, void *out_stack, int plane_w, const uint8_t *mask) {
    NhwcP p{};
    p.B = B; p.C = C; p.HW = HW; p.plane_w = plane_w; p.count = count ? 1 : 0;
    p.ct = (C + kTC - 1) / kTC;
    p.G = 1;
    if (HW >= kTP) {
        // as few tiles as hold the plane, of nearly the same size: what a short last tile leaves empty is spread over whole warps
        p.pt = (HW + kTP - 1) / kTP;
        p.P = ((HW + p.pt - 1) / p.pt + V - 1) / V * V;
    } else {
        // whole images, as many as fit and as leave two tiles per SM
        p.pt = 1;
        p.P = HW;
        const long long spread = static_cast<long long>(B) * p.ct / (2 * ctx->sm_count);
        p.G = kTP / HW;
        if (p.G > spread) p.G = spread > 1 ? static_cast<int>(spread) : 1;
    }
    const long long ntiles = static_cast<long long>((B + p.G - 1) / p.G) * p.ct * p.pt;
    p.ntiles = static_cast<int>(ntiles);
    const long long cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM, blocks = ntiles < cap ? ntiles : cap;
    p.step_p = static_cast<int>(blocks % p.pt);
    p.step_c = static_cast<int>(blocks / p.pt % p.ct);
    p.step_b = static_cast<int>(blocks / p.pt / p.ct);
    // (positions, channels, groups of images) -> distances
    auto far = [&](long long np, long long nc, long long nb) {
        const long long pitch = (C + 7) & ~7, e = np * p.P + nc * kTC * HW + nb * p.G * C * HW;
        return NhwcP::Far{e, np * p.P * pitch + nc * kTC + nb * p.G * HW * pitch, nc * kTC + nb * p.G * (HW + plane_w) * static_cast<long long>(C),
                          static_cast<unsigned long long>(e / 2) * kGamma};
    };
    p.far = far(p.step_p, p.step_c, p.step_b);
    p.wrap_p = far(-p.pt, 1, 0);
    p.wrap_c = far(0, -p.ct, 1);
    auto go = [&](auto kern) {
        return launch_chained(kern, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream,
                              static_cast<const T *>(delta), p, seed, step, static_cast<unsigned short *>(out),
                              static_cast<unsigned short *>(out_stack), ctx->state, static_cast<const unsigned char *>(mask));
    };
    if constexpr (sizeof(T) == 4) {
        if (mask != nullptr) return out_stack ? go(quantize_nhwc_kernel<T, V, true, true>) : go(quantize_nhwc_kernel<T, V, false, true>);
    }
    return out_stack ? go(quantize_nhwc_kernel<T, V, true, false>) : go(quantize_nhwc_kernel<T, V, false, false>);
}

// Planes of any size and channels of any number: a channel's row of the tile is covered by the aligned vectors that touch it
// (one more than a row holds), and what lies outside the row is dropped.
template <typename T, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_nhwc_any_kernel(const T *__restrict__ x, int B, int C, int HW, unsigned long long seed, const StepSource step,
                         unsigned short *__restrict__ out, DeviceState *__restrict__ st, int count,
                         const unsigned char *__restrict__ mask) {
    __shared__ __align__(16) unsigned char tile[2][kTileBytes];
    constexpr int V = Vec<T>::V;
    const unsigned ct = (C + kTC - 1) / kTC, pt = (HW + kTP - 1) / kTP, per_img = ct * pt, ntiles = B * per_img;
    const int pitch = (C + 7) & ~7;
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned nnz = 0, sat = 0, nz2 = 0;
    int buf = 0;
    for (unsigned t = blockIdx.x; t < ntiles; t += gridDim.x, buf ^= 1) {
        unsigned char *tl = tile[buf];
        const int b = t / per_img, rem = t - b * per_img, c0 = (rem / pt) * kTC, p0 = (rem - rem / pt * pt) * kTP;
        {
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
                unsigned long long u[V / 2];
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
                dithers_of<V>(e0, seed, u);
                decide<V>(v, u, inv, f, sat);
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (pp + j >= 0 && pp + j < len) {
                        nnz += f[j] != 0.f;
                        *reinterpret_cast<unsigned short *>(tl + tile_off<8>(pp + j, c)) = static_cast<unsigned short>(__float_as_uint(f[j]) >> 16);
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
                    *reinterpret_cast<const uint4 *>(tl + tile_off<8>(pp, ch * 8));
        }
        // the other buffer is written next; this one again only after the next barrier
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
    }
    nnz += pairs_total(nz2);
    if (count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}

// ---------------------------------------------------------------- bf16 planes of odd sizes
// Planes whose size is no multiple of 4 (7 x 7, 9 x 9, rows of 875 outputs, ...) written at a pitch that is a multiple of 8: the
// codes of eight consecutive elements then belong to unaligned places of one or two planes. A block takes 4096 consecutive
// elements, quantizes them with whole-vector loads as everywhere and keeps the codes as they come in shared memory; the output's
// 16-byte words that start among the first 4088 are put together from them (five 32-bit words each, shifted by half of one where
// a word starts on an odd element) and leave as one contiguous run. The last eight elements are the next run's first: it counts
// them. (The padding of a plane is never read by anybody.) Whole planes to a run, and planes of more than 784 elements and odd
// numbers of them code by code, before: 34 M elements of 53 x 53 planes 80 us.
constexpr int kRowRun = kThreads * kPerThread, kRowStep = kRowRun - 8;

template <typename T, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_rows_kernel(const T *__restrict__ x, long long n, int hw, int words, unsigned long long seed, const StepSource step,
                     unsigned short *__restrict__ out, DeviceState *__restrict__ st, int count, const unsigned char *__restrict__ mask) {
    constexpr int V = Vec<T>::V, NV = kPerThread / V, kBetween = kThreads * V;
    constexpr unsigned long long kBetweenZ = kBetween / 2 * kGamma;
    __shared__ __align__(16) unsigned run_s[2][kRowRun / 2 + 8];
    const long long nruns = (n + kRowStep - 1) / kRowStep;
    const bool counts_last = static_cast<int>(threadIdx.x) * V + (NV - 1) * kBetween < kRowStep;      // its last vector is not the next run's
    uint4 raw[NV];
    unsigned msk[MASKED ? NV : 1];
    unsigned long long u[NV][V / 2];
    auto load = [&](long long r) {
        const long long e = r * kRowStep + threadIdx.x * V;
        if (r * kRowStep + kRowRun <= n) {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                raw[k] = Vec<T>::raw(x + e + k * kBetween);
                if (MASKED) msk[k] = mask_word(mask, e + k * kBetween);
            }
        } else {
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                raw[k] = load_edge(x + e + k * kBetween, n - e - k * kBetween);
                if (MASKED) {
                    msk[k] = 0u;
                    for (int j = 0; j < V && e + k * kBetween + j < n; ++j) msk[k] |= static_cast<unsigned>(__ldg(mask + e + k * kBetween + j)) << (8 * j);
                }
            }
        }
    };
    long long r = blockIdx.x;
    unsigned long long z = counter_of(r * kRowStep + threadIdx.x * V, seed);
    const unsigned long long stride_z = static_cast<unsigned long long>(gridDim.x) * (kRowStep / 2) * kGamma;
    auto draw = [&]() {
#pragma unroll
        for (int k = 0; k < NV; ++k) dithers_at<V>(z + k * kBetweenZ, u[k]);
    };
    load(r);
    draw();
    keep_here(u);
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned sat = 0, nz2 = 0, nnz = 0;
    const int q_plane = kThreads / words, r_word = kThreads - q_plane * words;      // 16-byte words of the output: from a thread's one to its next
    const int next_rel = q_plane * hw + 8 * r_word, wrap_rel = hw - 8 * words;
    for (int buf = 0; r < nruns; buf ^= 1) {
        const long long here = r * kRowStep;
        unsigned short *const run = reinterpret_cast<unsigned short *>(run_s[buf]);
        unsigned h[NV][V / 2], top = 0u;
        const unsigned before = nz2;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            float v[V];
            Vec<T>::values(raw[k], v);
            if (MASKED) apply_mask(msk[k], v);
            quick_codes<V>(v, u[k], inv, h[k], top);
            if (k < NV - 1 || counts_last) count_pairs<V>(h[k], nz2);
        }
        if (needs_care(top)) {                                         // rare: clip, count, NaN
            nz2 = before;
#pragma unroll
            for (int k = 0; k < NV; ++k) {
                float v[V];
                unsigned long long d[V / 2];
                unsigned mc[V], clipped = 0u;
                Vec<T>::values(raw[k], v);
                if (MASKED) apply_mask(msk[k], v);
                dithers_at<V>(z + k * kBetweenZ, d);
                careful_codes<V>(v, d, inv, h[k], mc, clipped);
                if (k < NV - 1 || counts_last) {
                    sat += clipped;
                    count_pairs<V>(h[k], nz2);
                }
            }
        }
        r += gridDim.x;
        if (r < nruns) load(r);
#pragma unroll
        for (int k = 0; k < NV; ++k) store_vec<V>(run + threadIdx.x * V + k * kBetween, h[k]);
        z += stride_z;
        if (r < nruns) draw();
        __syncthreads();
        // the first output word that starts in the run, and this thread's
        long long plane, in_plane;
        split_index(here, hw, plane, in_plane);
        int w = (static_cast<int>(in_plane) + 7) >> 3, rel = 8 * w - static_cast<int>(in_plane);
        if (w == words) { w = 0; ++plane; rel = hw - static_cast<int>(in_plane); }
        uint4 *dst = reinterpret_cast<uint4 *>(out) + plane * words + w + threadIdx.x;
        const int skip = (w + static_cast<int>(threadIdx.x)) / words, w1 = w + static_cast<int>(threadIdx.x) - skip * words;
        const int end = static_cast<int>(n - here < kRowStep ? n - here : kRowStep);
        long long at = rel + static_cast<long long>(skip) * hw + 8 * (w1 - w);
        for (w = w1; at < end; dst += kThreads) {
            const int sh = (static_cast<int>(at) & 1) * 16;
            const unsigned *src = run_s[buf] + (at >> 1);
            const unsigned v0 = src[0], v1 = src[1], v2 = src[2], v3 = src[3], v4 = src[4];
            *dst = make_uint4(__funnelshift_r(v0, v1, sh), __funnelshift_r(v1, v2, sh), __funnelshift_r(v2, v3, sh), __funnelshift_r(v3, v4, sh));
            at += next_rel;
            w += r_word;
            if (w >= words) { w -= words; at += wrap_rel; }
        }
        // the other buffer is written next; this one again only after the next barrier
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
    }
    nnz += pairs_total(nz2);
    if (count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}

// Position-major planes of odd sizes: a run is a multiple of eight channels of one image, so that it starts on a 16-byte boundary
// and on an even element (the last run of an image has what is left; at 472 channels of 5x5 planes runs of eight, the only number
// that divides them, took 34 us for 1.4 M elements); its codes are kept as they come in whole words of shared memory, and eight
// channels of a position are eight 16-bit reads, a plane apart (in different banks for odd planes). Placing the codes one by one took 52 instructions an element.
constexpr int kOddElems = 6272;                   // most elements of a run

struct NhwcOut {
    int C;                        // channels: a multiple of 8
    unsigned short *stack;        // the copy with rows of zeros after every image (may be null)
    int plane_w;                  // how many
};

template <typename T, bool MASKED>
__global__ void __launch_bounds__(kThreads, kBlocksPerSM)
quantize_planes_odd_kernel(const T *__restrict__ x, long long nplanes, int hw, int per_run,
                           unsigned long long seed, const StepSource step, unsigned short *__restrict__ out,
                           DeviceState *__restrict__ st, int count, const unsigned char *__restrict__ mask, const NhwcOut nhwc) {
    constexpr int V = Vec<T>::V;
    // Vectors in hand per thread. 16 elements of fp32 spill 68 bytes (132 with a mask): calls of 64 -> 64 at 27x27, batch 128, take 83.6
    // us with them and 80.1 with eight (masked 89.7, 83.1); 64 -> 512 at 5x5, batch 300, 66.0 and 61.7 (71.7, 63.9)
    constexpr int NV = (V == 4 ? kPerThread / 2 : kPerThread) / V;
    constexpr int kBetween = kThreads * V;
    constexpr unsigned long long kBetweenZ = kBetween / 2 * kGamma;
    __shared__ __align__(16) unsigned run_s[kOddElems / 2 + 8];
    // a run's channels are of one image, whose last run has what is left of them
    const int per_image = (nhwc.C + per_run - 1) / per_run;
    const long long nruns = nplanes / nhwc.C * per_image;
    uint4 raw[NV];
    unsigned msk[MASKED ? NV : 1];
    unsigned long long u[NV][V / 2];
    // the run's elements from e on that this thread holds: those of its vectors that lie before the run's end
    auto load = [&](long long e, int left) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            raw[k] = k * kBetween < left ? Vec<T>::raw(x + e + k * kBetween) : make_uint4(0u, 0u, 0u, 0u);
            if (MASKED) msk[k] = k * kBetween < left ? mask_word(mask, e + k * kBetween) : 0u;
        }
    };
    auto draw = [&](unsigned long long zz) {
#pragma unroll
        for (int k = 0; k < NV; ++k) dithers_at<V>(zz + k * kBetweenZ, u[k]);
    };
    long long r = blockIdx.x, base = 0, image = 0;
    int c0 = 0, chans = 0, image_n = 0, c0_n = 0, chans_n = 0;       // the run in hand, and the next one
    // run r's first element and its length (a multiple of 8)
    auto find = [&]() {
        image_n = static_cast<int>(r / per_image);
        c0_n = static_cast<int>(r - static_cast<long long>(image_n) * per_image) * per_run;
        chans_n = nhwc.C - c0_n < per_run ? nhwc.C - c0_n : per_run;
        base = (static_cast<long long>(image_n) * nhwc.C + c0_n) * hw;
        return chans_n * hw;
    };
    int len = find(), done = threadIdx.x * V;                // elements of the run; the thread's place in it
    const unsigned long long tid_z = counter_of(done, seed);
    unsigned long long z = tid_z + static_cast<unsigned long long>(base / 2) * kGamma;
    load(base + done, len - done);
    draw(z);
    keep_here(u);
    const StepSource from = step_ahead(step);
    chain_wait();
    chain_release();
    const float delta = step_of<kThreads>(from, st);
    const float inv = delta > 0.f ? __fdiv_rn(1.0f, delta) : 0.f;      // Delta = 0: every code 0
    unsigned sat = 0, nz2 = 0, nnz = 0;
    int words = 1, q_pos = 0, r_word = 0, first_pos = 0, first_word = 0;      // 16-byte words of a position
    while (r < nruns) {
        const long long here = base;
        const int now = len;
        image = image_n;
        c0 = c0_n;
        if (chans != chans_n) {
            chans = chans_n;
            words = chans / 8;
            q_pos = kThreads / words;
            r_word = kThreads - q_pos * words;
            first_pos = threadIdx.x / words;
            first_word = threadIdx.x - first_pos * words;
        }
        // the run in rounds of NV vectors per thread; after its last one the next run's first is on its way
        while (true) {
            unsigned h[NV][V / 2], top = 0u;
            const unsigned before = nz2;
            const int at = done, left = now - at;
            const unsigned long long zz = z;
            if (left > 0) {
#pragma unroll
                for (int k = 0; k < NV; ++k) {
                    float v[V];
                    Vec<T>::values(raw[k], v);
                    if (MASKED) apply_mask(msk[k], v);
                    quick_codes<V>(v, u[k], inv, h[k], top);
                    count_pairs<V>(h[k], nz2);
                }
            }
            done += NV * kBetween;
            z += NV * kBetweenZ;
            const bool last = done - static_cast<int>(threadIdx.x) * V >= now;       // uniform
            if (last) {
                r += gridDim.x;
                len = r < nruns ? find() : 0;
                done = threadIdx.x * V;
                z = tid_z + static_cast<unsigned long long>(base / 2) * kGamma;
            }
            load(base + done, len - done);
            if (needs_care(top)) {                                  // rare: clip, count, NaN
                nz2 = before;
#pragma unroll 1
                for (int k = 0; k < NV; ++k) {
                    if (k * kBetween >= left) break;
                    float v[V];
                    unsigned long long d[V / 2];
                    unsigned hc[V / 2], mc[V];
                    Vec<T>::values(Vec<T>::raw(x + here + at + k * kBetween), v);
                    if (MASKED) apply_mask(mask_word(mask, here + at + k * kBetween), v);
                    dithers_at<V>(zz + k * kBetweenZ, d);
                    careful_codes<V>(v, d, inv, hc, mc, sat);
                    count_pairs<V>(hc, nz2);
                    store_vec<V>(reinterpret_cast<unsigned short *>(run_s) + at + k * kBetween, hc);
                }
            } else {
#pragma unroll
                for (int k = 0; k < NV; ++k)
                    if (k * kBetween < left) store_vec<V>(reinterpret_cast<unsigned short *>(run_s) + at + k * kBetween, h[k]);
            }
            if (last) break;
            if (done < now) draw(z);
        }
        __syncthreads();
        const int tall = hw + (nhwc.stack ? nhwc.plane_w : 0);
        unsigned short *dst = out + image * hw * nhwc.C + c0, *to = nhwc.stack + image * tall * nhwc.C + c0;
        const unsigned short *src = reinterpret_cast<const unsigned short *>(run_s);
        int pp = first_pos, w = first_word;
        for (int i = threadIdx.x; i < tall * words; i += kThreads) {
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (pp < hw) {
                unsigned k[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) k[j] = src[(8 * w + j) * hw + pp];
                v = make_uint4(__byte_perm(k[0], k[1], 0x5410), __byte_perm(k[2], k[3], 0x5410), __byte_perm(k[4], k[5], 0x5410),
                               __byte_perm(k[6], k[7], 0x5410));
                *reinterpret_cast<uint4 *>(dst + static_cast<long long>(pp) * nhwc.C + 8 * w) = v;
            }
            if (nhwc.stack != nullptr) *reinterpret_cast<uint4 *>(to + static_cast<long long>(pp) * nhwc.C + 8 * w) = v;
            pp += q_pos;
            w += r_word;
            if (w >= words) { w -= words; ++pp; }
        }
        if (nz2 & 0x80008000u) { nnz += pairs_total(nz2); nz2 = 0; }
        if (r >= nruns) break;
        draw(z);
        __syncthreads();                                            // the buffer is written again
    }
    nnz += pairs_total(nz2);
    if (count) publish_counts<kThreads>(nnz, delta > 0.f ? sat : 0u, st, nullptr);
}
template <typename T>
int run_planes_odd(dbp_ctx *ctx, const void *delta, long long B, int hw, int per_run, unsigned long long seed, const StepSource &step,
                   void *out, bool count, const uint8_t *mask, const NhwcOut &nhwc) {
    const long long nruns = B * ((nhwc.C + per_run - 1) / per_run), cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM;
    auto go = [&](auto kern) {
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(nruns < cap ? nruns : cap)), dim3(kThreads), 0, ctx->stream,
                                      static_cast<const T *>(delta), B * nhwc.C, hw, per_run, seed, step, static_cast<unsigned short *>(out),
                                      ctx->state, count ? 1 : 0, static_cast<const unsigned char *>(mask), nhwc));
    };
    if constexpr (sizeof(T) == 4) {
        if (mask != nullptr) return go(quantize_planes_odd_kernel<T, true>);
    }
    return go(quantize_planes_odd_kernel<T, false>);
}

// Channels in a run of the position-major form: as many as fit, at most 64 (a row of the output), but fewer (not below 16: 32 bytes
// of a row) where the runs would not cover the SMs twice. 0: eight do not fit.
int odd_channels_per_run(long long B, int C, int hw, int sms) {
    int n = kOddElems / hw / 8 * 8;
    if (n > 64) n = 64;
    while (n > 16 && B * ((C + n - 1) / n) < 2ll * sms) n -= 8;
    return n;
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
    if ((dense != nullptr) == (planes != nullptr)) return DBP_EINVAL;          // one form a call
    // rows of the output start on 16-byte boundaries
    if (planes != nullptr && pitch != hw && (hw <= 0 || hw >= (1 << 30) || numel % hw != 0 || pitch != (hw + 7) / 8 * 8)) return DBP_EINVAL;
    if (planes != nullptr && pitch != hw && (hw & 3) != 0) {
        const long long nruns = (numel + kRowStep - 1) / kRowStep, most = static_cast<long long>(ctx->sm_count) * kBlocksPerSM;
        auto rows = [&](auto kern, auto x) {
            return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(nruns < most ? nruns : most)), dim3(kThreads), 0, ctx->stream, x, numel,
                                          static_cast<int>(hw), static_cast<int>(pitch / 8), seed, step, planes, ctx->state, count ? 1 : 0, m));
        };
        return dtype != DBP_F32 ? rows(quantize_rows_kernel<__nv_bfloat16, false>, xb)
               : m              ? rows(quantize_rows_kernel<float, true>, xf)
                                : rows(quantize_rows_kernel<float, false>, xf);
    }
    constexpr int kTile = kThreads * kPerThread;
    long long blocks = (numel / v * v + kTile - 1) / kTile;
    if (blocks < 1) blocks = 1;
    const long long cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM;
    if (blocks > cap) blocks = cap;
    CodeSinks out{};
    out.dense8 = dense;
    out.planes16 = planes;
    out.hw = hw > 0 ? hw : 1;
    out.pitch = pitch > 0 ? pitch : 1;
    out.count = count ? 1 : 0;
    const long long between = kThreads * v, next = blocks * kTile - (kTile - between);
    out.rest1 = static_cast<int>(between % out.hw);
    out.rest2 = static_cast<int>(next % out.hw);
    out.dist1 = between / out.hw * out.pitch + out.rest1;
    out.dist2 = next / out.hw * out.pitch + out.rest2;
    const int sink = dense ? kBytes : out.pitch == out.hw ? kSame : kPad4;
    auto go = [&](auto kern, auto x) {
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(blocks)), dim3(kThreads), 0, ctx->stream, x, numel, seed, step, out,
                                      ctx->state, m));
    };
    auto pick = [&](auto s) {
        constexpr int S = decltype(s)::value;
        return dtype != DBP_F32 ? go(quantize_dense_kernel<__nv_bfloat16, false, S>, xb)
               : m              ? go(quantize_dense_kernel<float, true, S>, xf)
                                : go(quantize_dense_kernel<float, false, S>, xf);
    };
    if (step.late) {                             // fp32 gradients of 5x5 layers, whole vectors, one byte per element
        if (sink != kBytes || dtype != DBP_F32 || numel % 4 != 0) return DBP_EINVAL;
        return m ? go(quantize_dense_kernel<float, true, kBytes, true>, xf) : go(quantize_dense_kernel<float, false, kBytes, true>, xf);
    }
    switch (sink) {
        case kBytes: return pick(std::integral_constant<int, kBytes>());
        case kSame: return pick(std::integral_constant<int, kSame>());
        default: return pick(std::integral_constant<int, kPad4>());
    }
}

// delta_z [B][C][HW] -> bf16 codes [B][HW][C rounded up to a multiple of 8]
int launch_quantize_nhwc(dbp_ctx *ctx, const void *delta, int dtype, long long B, long long C, long long HW,
                         unsigned long long seed, const StepSource &step, void *codes_nhwc, bool count,
                         void *codes_stack, int plane_w, const uint8_t *mask) {
    if (B * C * HW >= (1ll << 40) || HW >= (1ll << 25)) return DBP_EUNSUPPORTED;
    if (B * ((C + kTC - 1) / kTC) * ((HW + kTP - 1) / kTP) >= (1ll << 31)) return DBP_EUNSUPPORTED;
    if (mask != nullptr && dtype != DBP_F32) return DBP_EUNSUPPORTED;
    // the stacked copy is written by the paths for planes smaller than a tile; the rows of image b start at
    // b (HW + W) however many images make up a tall image: the stacking only adds the zero rows
    if (codes_stack != nullptr && (HW >= kTP || C % 8 != 0 || plane_w <= 0 || HW + plane_w > kTP)) return DBP_EINVAL;
    const int b = static_cast<int>(B), c = static_cast<int>(C), hw = static_cast<int>(HW);
    if (hw % 4 == 0) {
        auto run = [&](auto kern) { return cuda_ok(kern(ctx, delta, b, c, hw, seed, step, codes_nhwc, count, codes_stack, plane_w, mask)); };
        return dtype == DBP_F32 ? run(run_nhwc<float, 4>) : hw % 8 == 0 ? run(run_nhwc<__nv_bfloat16, 8>) : run(run_nhwc<__nv_bfloat16, 4>);
    }
    if (c % 8 == 0) {
        if (const int n = odd_channels_per_run(B, c, hw, ctx->sm_count)) {
            const NhwcOut nh{c, static_cast<unsigned short *>(codes_stack), plane_w};
            return dtype != DBP_F32 ? run_planes_odd<__nv_bfloat16>(ctx, delta, B, hw, n, seed, step, codes_nhwc, count, mask, nh)
                                    : run_planes_odd<float>(ctx, delta, B, hw, n, seed, step, codes_nhwc, count, mask, nh);
        }
    }
    const long long ntiles = B * ((C + kTC - 1) / kTC) * ((HW + kTP - 1) / kTP), cap = static_cast<long long>(ctx->sm_count) * kBlocksPerSM;
    auto go = [&](auto kern, auto x) {
        return cuda_ok(launch_chained(kern, dim3(static_cast<unsigned>(ntiles < cap ? ntiles : cap)), dim3(kThreads), 0, ctx->stream, x, b, c,
                                      hw, seed, step, static_cast<unsigned short *>(codes_nhwc), ctx->state, count ? 1 : 0,
                                      static_cast<const unsigned char *>(mask)));
    };
    const float *xf = static_cast<const float *>(delta);
    return dtype != DBP_F32 ? go(quantize_nhwc_any_kernel<__nv_bfloat16, false>, static_cast<const __nv_bfloat16 *>(delta))
           : mask           ? go(quantize_nhwc_any_kernel<float, true>, xf)
                            : go(quantize_nhwc_any_kernel<float, false>, xf);
}

}  // namespace dbp
