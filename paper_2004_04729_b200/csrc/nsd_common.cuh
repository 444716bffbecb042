// The NSD decision (Algorithm 1, Eq. (nsd)) as every quantizer kernel takes it: dither from the SplitMix64 counter
// sequence, q = floor(x / Delta + u) in fp32, clipped and counted.
#pragma once

#include "dbp_internal.cuh"

namespace dbp {
namespace nsd {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kGamma = 0x9E3779B97F4A7C15ull;
constexpr float kMagic = 12582912.0f;             // 1.5 * 2^23: a float in [2^23, 2^24) has unit spacing
constexpr float kDitherShift = -0.99999994f;      // 2^-24 - 1

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// ---- two fp32 operations per instruction
__device__ __forceinline__ unsigned long long pack2(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long r, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ unsigned long long add2(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long add2_down(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// largest magnitude of three; NaN if one of them is
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// The dithers of the pair of elements that shares output number c = z / gamma of the sequence: u = (2k+1) 2^-24 from the
// top 23 bits k of the output's halves, low half first. The output is z ^ (z >> 31) of the mixed z: of its high half
// that xor only changes bit 0, of its low half it is bits 0-30 of (high half << 1) (and bit 31's neighbour in bit 0), so
// the 23 bits that count need neither 64-bit shift. 1 + k 2^-23 is one funnel shift, and u that plus 2^-24 - 1.
// Written in 32-bit halves, a 64-bit product as three multiply-adds: 11.5 instructions an element against 12.5 from 64-bit
// expressions. Shifts, xors and byte permutations issue every second clock of a scheduler, on one pipe, multiplications
// every second clock on another (wide ones every fourth), additions every clock. The draw takes 16.8 clocks an element (14 of
// the first pipe), the whole decision 22, whether two or eight warps per scheduler run. Multiplications in place of shifts, or
// mixed-precision additions in place of the conversion from bf16, are no faster.
// SHORT: for a kernel that is a chain of latencies and not of instructions, a product is the sum of two independent ones: one
// instruction more, one less behind another (a small linear layer's call 9.43 against 9.51 us; the thin 1x1 call 73.9 against 71.9).
template <bool SHORT>
__device__ __forceinline__ void mul_low64(unsigned &lo, unsigned &hi, unsigned clo, unsigned chi) {
    if (SHORT) {
        asm("{\n\t.reg .u64 p;\n\t.reg .u32 a, b, h;\n\t"
            "mul.lo.u32 h, %0, %3;\n\t"
            "mad.lo.u32 h, %1, %2, h;\n\t"
            "mul.wide.u32 p, %0, %2;\n\t"
            "mov.b64 {a, b}, p;\n\t"
            "add.u32 %1, b, h;\n\t"
            "mov.b32 %0, a;\n\t}"
            : "+r"(lo), "+r"(hi) : "r"(clo), "r"(chi));
    } else {
        asm("{\n\t.reg .u64 p;\n\t.reg .u32 a, b, h;\n\t"
            "mul.wide.u32 p, %0, %2;\n\t"
            "mov.b64 {a, b}, p;\n\t"
            "mad.lo.u32 h, %0, %3, b;\n\t"
            "mad.lo.u32 %1, %1, %2, h;\n\t"
            "mov.b32 %0, a;\n\t}"
            : "+r"(lo), "+r"(hi) : "r"(clo), "r"(chi));
    }
}
template <bool SHORT = false>
__device__ __forceinline__ unsigned long long dither2(unsigned long long z) {
    unsigned lo = static_cast<unsigned>(z), hi = static_cast<unsigned>(z >> 32);
    lo ^= __funnelshift_r(lo, hi, 30);
    hi ^= hi >> 30;
    mul_low64<SHORT>(lo, hi, 0x1CE4E5B9u, 0xBF58476Du);
    lo ^= __funnelshift_r(lo, hi, 27);
    hi ^= hi >> 27;
    mul_low64<SHORT>(lo, hi, 0x133111EBu, 0x94D049BBu);
    lo ^= hi + hi;
    return add2(pack2(__uint_as_float(__funnelshift_r(lo, 0x7fu, 9)), __uint_as_float(__funnelshift_r(hi, 0x7fu, 9))),
                pack2(kDitherShift, kDitherShift));
}
__device__ __forceinline__ unsigned long long counter_of(long long e, unsigned long long seed) {      // e even
    return seed + (static_cast<unsigned long long>(e >> 1) + 1ull) * kGamma;
}
// dithers of V elements whose first pair has the counter z, pairs packed
template <int V, bool SHORT = false>
__device__ __forceinline__ void dithers_at(unsigned long long z, unsigned long long (&u)[V / 2]) {
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        u[j] = dither2<SHORT>(z);
        z += kGamma;
    }
}
// and of V elements whose first has the even index e0
template <int V, bool SHORT = false>
__device__ __forceinline__ void dithers_of(long long e0, unsigned long long seed, unsigned long long (&u)[V / 2]) {
    dithers_at<V, SHORT>(counter_of(e0, seed), u);
}
// Dithers drawn ahead of a wait stay there: without this the compiler moves the arithmetic behind the wait (about 1 us of each
// of the quantizers).
template <int N, int P>
__device__ __forceinline__ void keep_here(unsigned long long (&u)[N][P]) {
#pragma unroll
    for (int k = 0; k < N; ++k)
#pragma unroll
        for (int j = 0; j < P; ++j) asm volatile("" : "+l"(u[k][j]));
}
// careful decision: clipped to [-127, 127], clipped codes counted, NaN gives 0. Returns the bits of kMagic + code (the
// low byte is the code's two's-complement byte).
__device__ __forceinline__ unsigned careful_bits(float x, float inv, float u, unsigned &sat) {
    const float t = __fmaf_rn(x, inv, u);
    const float tc = fminf(fmaxf(t, -127.f), 127.99999f);
    const bool num = (t == t);
    sat += (num && tc != t) ? 1u : 0u;
    return num ? __float_as_uint(__fadd_rd(tc, kMagic)) : __float_as_uint(kMagic);
}
// Codes of V elements as floats (exact small integers). The common case (every |x / Delta + u| <= 127, no NaN) needs no
// clamp: floor(t) is the round-down sum with kMagic, less kMagic.
template <int V>
__device__ __forceinline__ void decide(const float (&x)[V], const unsigned long long (&u)[V / 2], float inv, float (&f)[V], unsigned &sat) {
    const unsigned long long inv2 = pack2(inv, inv), up = pack2(kMagic, kMagic), down = pack2(-kMagic, -kMagic);
    float top = 0.f;
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        const unsigned long long t = fma2(pack2(x[2 * j], x[2 * j + 1]), inv2, u[j]);
        float a, b;
        unpack2(t, a, b);
        top = max3_abs(a, b, top);
        unpack2(add2(add2_down(t, up), down), f[2 * j], f[2 * j + 1]);
    }
    if (!(top <= 127.f)) {                          // rare: clip, count, NaN
#pragma unroll
        for (int j = 0; j < V; ++j) {
            float ua, ub;
            unpack2(u[j >> 1], ua, ub);
            f[j] = __uint_as_float(careful_bits(x[j], inv, (j & 1) ? ub : ua, sat)) - kMagic;
        }
    }
}
// the codes as bf16, two to a word: an integer of at most 8 bits is exact in bf16, which is the float's upper half
template <int V>
__device__ __forceinline__ void pack_bf16(const float (&f)[V], unsigned (&h)[V / 2]) {
#pragma unroll
    for (int j = 0; j < V / 2; ++j) h[j] = __byte_perm(__float_as_uint(f[2 * j]), __float_as_uint(f[2 * j + 1]), 0x7632);
}
// The same without a branch, for code that decides several vectors and looks once whether one of them needs the careful
// decision: codes as packed bf16 words (h) and as the low bytes of m, and in `top` the largest magnitude seen in either half
// of a word (a sign and NaN included). A code out of range shows there as 128 or more, whatever the sum with kMagic made of
// it. What is not used of h or m costs nothing.
template <int V>
__device__ __forceinline__ void quick_codes(const float (&x)[V], const unsigned long long (&u)[V / 2], float inv, unsigned (&h)[V / 2],
                                            unsigned (&m)[V], unsigned &top) {
    const unsigned long long inv2 = pack2(inv, inv), up = pack2(kMagic, kMagic), down = pack2(-kMagic, -kMagic);
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        const unsigned long long t = add2_down(fma2(pack2(x[2 * j], x[2 * j + 1]), inv2, u[j]), up);
        float a, b;
        unpack2(t, a, b);
        m[2 * j] = __float_as_uint(a);
        m[2 * j + 1] = __float_as_uint(b);
        unpack2(add2(t, down), a, b);
        h[j] = __byte_perm(__float_as_uint(a), __float_as_uint(b), 0x7632);
        asm("max.NaN.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(top) : "r"(h[j]));
    }
}
template <int V>
__device__ __forceinline__ void quick_codes(const float (&x)[V], const unsigned long long (&u)[V / 2], float inv, unsigned (&h)[V / 2],
                                            unsigned &top) {
    unsigned m[V];
    quick_codes<V>(x, u, inv, h, m, top);
}
// the same for the same elements of two rows: a word holds the codes of one place, row a's in its low half
template <int V>
__device__ __forceinline__ void quick_codes2(const float (&xa)[V], const float (&xb)[V], const unsigned long long (&ua)[V / 2],
                                             const unsigned long long (&ub)[V / 2], float inv, unsigned (&w)[V], unsigned &top) {
    const unsigned long long inv2 = pack2(inv, inv), up = pack2(kMagic, kMagic), down = pack2(-kMagic, -kMagic);
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        float a0, a1, b0, b1;
        unpack2(add2(add2_down(fma2(pack2(xa[2 * j], xa[2 * j + 1]), inv2, ua[j]), up), down), a0, a1);
        unpack2(add2(add2_down(fma2(pack2(xb[2 * j], xb[2 * j + 1]), inv2, ub[j]), up), down), b0, b1);
        w[2 * j] = __byte_perm(__float_as_uint(a0), __float_as_uint(b0), 0x7632);
        w[2 * j + 1] = __byte_perm(__float_as_uint(a1), __float_as_uint(b1), 0x7632);
        asm("max.NaN.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(top) : "r"(w[2 * j]));
        asm("max.NaN.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(top) : "r"(w[2 * j + 1]));
    }
}
__device__ __forceinline__ bool needs_care(unsigned top) {            // 0x42fe: 127
    return __vmaxu2(top & 0x7fff7fffu, 0x42fe42feu) != 0x42fe42feu;
}
template <int V>
__device__ __forceinline__ void careful_codes(const float (&x)[V], const unsigned long long (&u)[V / 2], float inv, unsigned (&h)[V / 2],
                                              unsigned (&m)[V], unsigned &sat) {
#pragma unroll
    for (int j = 0; j < V / 2; ++j) {
        float ua, ub;
        unpack2(u[j], ua, ub);
        m[2 * j] = careful_bits(x[2 * j], inv, ua, sat);
        m[2 * j + 1] = careful_bits(x[2 * j + 1], inv, ub, sat);
        h[j] = __byte_perm(__float_as_uint(__uint_as_float(m[2 * j]) - kMagic), __float_as_uint(__uint_as_float(m[2 * j + 1]) - kMagic),
                           0x7632);
    }
}
// the bytes of such sums, four to a word in element order
template <int V>
__device__ __forceinline__ void low_bytes(const unsigned (&m)[V], unsigned (&pk)[V / 4]) {
#pragma unroll
    for (int w = 0; w < V / 4; ++w)
        pk[w] = __byte_perm(__byte_perm(m[4 * w], m[4 * w + 1], 0x0040), __byte_perm(m[4 * w + 2], m[4 * w + 3], 0x0040), 0x5410);
}
// non-zero codes of the even and of the odd elements, counted in the halves of a word (a code's bf16 bits are zero only
// for code 0); add up to 65535 of each before reading it with `pairs_total`
template <int V>
__device__ __forceinline__ void count_pairs(const unsigned (&h)[V / 2], unsigned &nz2) {
#pragma unroll
    for (int j = 0; j < V / 2; ++j) nz2 += __vminu2(h[j], 0x00010001u);
}
__device__ __forceinline__ unsigned pairs_total(unsigned nz2) { return (nz2 & 0xffffu) + (nz2 >> 16); }

// ---- the elements of delta_z in 128-bit vectors
template <typename T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int V = 4;
    __device__ static uint4 raw(const float *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
    __device__ static void values(const uint4 &q, float (&v)[4]) {
        v[0] = __uint_as_float(q.x); v[1] = __uint_as_float(q.y); v[2] = __uint_as_float(q.z); v[3] = __uint_as_float(q.w);
    }
    __device__ static float one(const float *p) { return __ldg(p); }
};
template <>
struct Vec<__nv_bfloat16> {
    static constexpr int V = 8;
    __device__ static uint4 raw(const __nv_bfloat16 *p) { return __ldg(reinterpret_cast<const uint4 *>(p)); }
    __device__ static void values(const uint4 &q, float (&v)[8]) {
        const unsigned w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[2 * i] = __uint_as_float(w[i] << 16);            // bf16 -> fp32 is exact
            v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
        }
    }
    __device__ static float one(const __nv_bfloat16 *p) {
        return __uint_as_float(static_cast<unsigned>(__ldg(reinterpret_cast<const unsigned short *>(p))) << 16);
    }
};

// A vector that the tensor's end cuts: its first `left` elements, the others zero
template <typename T>
__device__ __forceinline__ uint4 load_edge(const T *p, long long left) {
    unsigned w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int j = 0; j < Vec<T>::V; ++j)
        if (j < left) {
            const unsigned b = __float_as_uint(Vec<T>::one(p + j));
            if (Vec<T>::V == 4) w[j] = b;
            else w[j / 2] |= j & 1 ? b : b >> 16;
        }
    return make_uint4(w[0], w[1], w[2], w[3]);
}

// ---- the step size
// Every CTA of a quantizer adds up the statistics kernel's partial sums by itself, in the same order, so all hold the
// same Delta: one L2 round trip at the head of the quantizer instead of an election of a last block, a fence, a ticket
// and two more round trips at the end of the statistics kernel (about 2 us of every call's chain).
// Delta = scale * sigma rounded once to fp32, sigma the population standard deviation about the mean; 0 (every code 0)
// for constant and for non-finite tensors. The first CTA publishes it. All threads of the block call this.
// Returns Delta, or 0 where no code can be non-zero.
// The parameters it needs, in registers: read ahead of the wait for the statistics kernel.
__device__ __forceinline__ StepSource step_ahead(StepSource s) {
    asm volatile("" : "+l"(s.partials), "+r"(s.nparts), "+f"(s.scale), "+d"(s.inv_numel), "+l"(s.given), "+l"(s.publish[0]),
                 "+l"(s.publish[1]), "+l"(s.publish[2]));
    return s;
}
template <int THREADS>
__device__ __forceinline__ float step_of(const StepSource &s, DeviceState *st) {
    __shared__ double sum_s[2][THREADS / 32];
    __shared__ float delta_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (s.given != nullptr) {
        const float d = __ldcg(s.given);
        if (blockIdx.x == 0 && threadIdx.x == 0)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (s.publish[i] != nullptr) *s.publish[i] = d;
        return d > 0.f && d < __int_as_float(0x7f800000) ? d : 0.f;
    }
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < s.nparts; i += THREADS) {
        const double2 v = __ldcg(reinterpret_cast<const double2 *>(s.partials) + i);
        a += v.x;
        b += v.y;
    }
    a = warp_sum(a);
    b = warp_sum(b);
    if (lane == 0) { sum_s[0][warp] = a; sum_s[1][warp] = b; }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = 0.0; b = 0.0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) { a += sum_s[0][w]; b += sum_s[1][w]; }
        float d = 0.f;
        if (!isfinite(a) || !isfinite(b)) {
            if (blockIdx.x == 0) st->nonfinite = 1;
        } else {
            const double mean = a * s.inv_numel;
            double var = b * s.inv_numel - mean * mean;
            if (var < 0.0) var = 0.0;
            d = static_cast<float>(static_cast<double>(s.scale) * sqrt(var));
        }
        if (blockIdx.x == 0)
#pragma unroll
            for (int i = 0; i < 3; ++i)
                if (s.publish[i] != nullptr) *s.publish[i] = d;
        delta_s = d;
    }
    __syncthreads();
    const float d = delta_s;
    return d > 0.f && d < __int_as_float(0x7f800000) ? d : 0.f;
}

// a block's counts to the context's counters (and a caller's): one atomic each
template <int THREADS>
__device__ __forceinline__ void publish_counts(unsigned nnz, unsigned sat, DeviceState *st, unsigned long long *nnz_out) {
    __shared__ unsigned cnt_s[2];
    if (threadIdx.x < 2) cnt_s[threadIdx.x] = 0u;
    __syncthreads();
    nnz = __reduce_add_sync(kFull, nnz);
    sat = __reduce_add_sync(kFull, sat);
    if ((threadIdx.x & 31) == 0) {
        if (nnz) atomicAdd(&cnt_s[0], nnz);
        if (sat) atomicAdd(&cnt_s[1], sat);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        if (cnt_s[0]) {
            atomicAdd(&st->nnz, static_cast<unsigned long long>(cnt_s[0]));
            if (nnz_out) atomicAdd(nnz_out, static_cast<unsigned long long>(cnt_s[0]));
        }
        if (cnt_s[1]) atomicAdd(&st->saturated, static_cast<unsigned long long>(cnt_s[1]));
    }
}

}  // namespace nsd
}  // namespace dbp
