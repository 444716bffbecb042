// Both products of a 5x5 layer of few channels (LeNet-5-like networks: stride 1, padding 2) in one launch, by fp32 FMAs on
// the dense codes:
//   dX[b,ci,y,x]    = Delta sum_{co,ky,kx} q[b,co,y-ky+2,x-kx+2] W[co,ci,ky,kx]
//   dW[co,ci,ky,kx] = Delta sum_{b,y,x}    q[b,co,y,x] X[b,ci,y+ky-2,x+kx-2]
// A handful of channels on either side fills a sixteenth of a tensor-core tile, and walking the non-zero codes (the gather
// kernels) keeps one lane per input channel busy; the multiply-adds of a whole image are a few microseconds of one SM's FMA
// pipe. So a CTA takes one image at a time, its codes, activations and the weights in shared memory with their zero
// borders, and both products come out of register tiles whose operands are 16-byte shared-memory loads:
//   dX: a thread owns 2 input channels x 4 columns; per (co, ky) two loads of codes, four of weights, 40 FMAs;
//   dW: a thread owns 4 output channels x 5 kernel columns of one (ci, ky) over a share of the image's rows; per four
//       columns two loads of activations, four of codes, 80 FMAs. Its sums stay in registers over the CTA's images; the
//       row shares are added in shared memory and the copy engine adds the CTA's block into dW (cleared before by the
//       statistics kernel; the order of the CTAs, hence the last bits of dW, can differ from run to run).
// LeNet-5-like, batch 128, fp32: second layer (6 -> 16 channels at 16x16, both products) 165 us on the gather kernels, 19 here
// with every value loaded and placed before the next; first layer (1 -> 6 at 32x32, dW) 111 us there, 11 here. Loaded ahead and
// placed in different banks the two are 12 us shorter in the chain of the network's kernels (61.9 -> 49.3 us in all; by themselves
// they are bound by the FMAs, 5 us of the second layer, and their start and end).
#include "tc_common.cuh"

namespace dbp {

namespace {

constexpr int kThreads5 = 512;
constexpr int kMaxFloats5 = 56 * 1024;             // shared memory of a CTA
constexpr int kHalfFloats5 = (228 / 2 - 1) * 256;  // and of one of two on an SM

struct Direct5P {
    const int8_t *codes;          // [B][Cout][H][W]
    const void *X, *W;
    const float *delta_p;
    float *dW;                    // null: not wanted
    void *dX;
    int B, Cin, Cout, H, Wd;
    int pitch;                    // floats per shared-memory row of an image with its border: W rounded up to 4, plus 4
    int plane;                    // floats per output channel of the codes with their border: an odd multiple of 4 where that fits
    int cop, co4;                 // output channels rounded up to 4, and a quarter of that
    int rg;                       // row shares of dW
};

__device__ __forceinline__ float value_of(float v) { return v; }
__device__ __forceinline__ float value_of(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ void store_value(float *p, float v) { *p = v; }
__device__ __forceinline__ void store_value(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

// What the whole CTA brings into shared memory: a thread's next U values are loaded before the first of them is placed. One by one
// each waited for its own trip to the L2: the codes of the second layer below were 3 us of this kernel, of the first 4.
template <int U, typename V, typename A, typename F>
__device__ __forceinline__ void each_of(int n, const V *src, A &&at, F &&place) {
#pragma unroll 1
    for (int i0 = threadIdx.x; i0 < n; i0 += U * kThreads5) {
        V v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * kThreads5 < n) v[u] = src[at(i0 + u * kThreads5)];
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (i0 + u * kThreads5 < n) place(i0 + u * kThreads5, v[u]);
    }
}

// CTAS: how many share an SM: two in half the registers, with two values in flight per thread in place of four or eight.
template <typename T, typename O, int CTAS>
__global__ void __launch_bounds__(kThreads5, CTAS)
direct5_kernel(const Direct5P p) {
    constexpr int U = CTAS == 2 ? 2 : 4, UB = CTAS == 2 ? 2 : 8;
    extern __shared__ __align__(16) float smem5[];
    const int tid = threadIdx.x;
    const int H = p.H, Wd = p.Wd, Wr = p.pitch - 4, Hp = H + 4, HW = H * Wd;
    const bool want_dx = p.dX != nullptr, want_dw = p.dW != nullptr;
    float *qa = smem5;                                               // [Cout][plane], rows of pitch: codes with a border of zeros (dX)
    float *w_s = qa + (want_dx ? p.Cout * p.plane : 0);         // [Cout][Cin rounded up to 2][5][8] (dX)
    const int cip = (p.Cin + 1) & ~1;
    float *qb = w_s + (want_dx ? p.Cout * cip * 40 : 0);             // [H][Wr][cop]: codes, channels innermost (dW)
    float *x_s = qb + (want_dw ? H * Wr * p.cop : 0);                // [Cin][H + 4][pitch]: activations with their border (dW)
    const int total = (want_dx ? p.Cout * (p.plane + cip * 40) : 0) + (want_dw ? H * Wr * p.cop + p.Cin * Hp * p.pitch : 0);

    // borders and padding stay zero; the inside is written for every image
    for (int i = tid; i < total / 4; i += kThreads5) reinterpret_cast<float4 *>(smem5)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    auto same = [](int i) { return i; };
    auto load_x = [&](int b) {
        const T *src = static_cast<const T *>(p.X) + static_cast<long long>(b) * p.Cin * HW;
        each_of<U>(p.Cin * HW, src, same, [&](int i, T v) {
            const int ci = i / HW, r = i - ci * HW, y = r / Wd, x = r - y * Wd;
            x_s[(ci * Hp + y + 2) * p.pitch + x + 2] = value_of(v);
        });
    };
    // the layer's inputs do not depend on the kernel before this one (the quantizer): they come in while it runs
    if (want_dx)
        each_of<U>(p.Cout * p.Cin * 25, static_cast<const T *>(p.W), same, [&](int i, T v) {
            const int t = i % 25, c = i / 25, co = c / p.Cin, ci = c - co * p.Cin;
            w_s[((co * cip + ci) * 5 + t / 5) * 8 + t % 5] = value_of(v);
        });
    if (want_dw) load_x(blockIdx.x);
    chain_wait();
    chain_release();
    const float delta = *p.delta_p;

    // dW: my four output channels, input channel, kernel row, share of the rows
    const int combos = p.co4 * p.Cin * 5;
    const int cmb = tid % combos, rg = tid / combos;
    const int q4 = cmb % p.co4, ky_w = (cmb / p.co4) % 5, ci_w = cmb / (p.co4 * 5);
    float acc_w[4][5];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 5; ++k) acc_w[j][k] = 0.f;

    for (int b = blockIdx.x; b < p.B; b += gridDim.x) {
        if (b != static_cast<int>(blockIdx.x)) {
            __syncthreads();                                         // the previous image has been used
            if (want_dw) load_x(b);
        }
        const int8_t *src = p.codes + static_cast<long long>(b) * p.Cout * HW;
        if ((Wd & 3) == 0) {
            // four codes of a row at a time, neighbouring threads on neighbouring channels: their words lie in different banks in
            // both copies (along a row they lay in two)
            const int quads = HW / 4, wq = Wd / 4;
            each_of<U>(p.Cout * quads, reinterpret_cast<const char4 *>(src), [&](int i) { return i % p.Cout * quads + i / p.Cout; }, [&](int i, char4 v) {
                const int r = i / p.Cout, co = i - r * p.Cout, y = r / wq, x = (r - y * wq) * 4;
                const float f[4] = {static_cast<float>(v.x), static_cast<float>(v.y), static_cast<float>(v.z), static_cast<float>(v.w)};
                float *const a = qa + co * p.plane + (y + 2) * p.pitch + x + 2, *const c = qb + (y * Wr + x) * p.cop + co;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (want_dx) a[k] = f[k];
                    if (want_dw) c[k * p.cop] = f[k];
                }
            });
        } else {
            each_of<UB>(p.Cout * HW, src, same, [&](int i, int8_t v) {
                const int co = i / HW, r = i - co * HW, y = r / Wd, x = r - y * Wd;
                const float f = static_cast<float>(v);
                if (want_dx) qa[co * p.plane + (y + 2) * p.pitch + x + 2] = f;
                if (want_dw) qb[(y * Wr + x) * p.cop + co] = f;
            });
        }
        __syncthreads();
        if (want_dx) {
            const int xt = Wr / 4, items = xt * H * (cip / 2);
            for (int it = tid; it < items; it += kThreads5) {
                const int x0 = (it % xt) * 4, r = it / xt, y = r % H, c2 = (r / H) * 2;
                float acc[2][4] = {};
                for (int co = 0; co < p.Cout; ++co) {
                    // code row y - ky + 2 lies at row y + 4 - ky of the bordered image, column x - kx + 2 at x - kx + 4
                    const float *q = qa + co * p.plane + y * p.pitch + x0;
                    const float *w = w_s + (co * cip + c2) * 40;
#pragma unroll
                    for (int ky = 0; ky < 5; ++ky) {
                        const float4 a = *reinterpret_cast<const float4 *>(q + (4 - ky) * p.pitch);
                        const float4 c = *reinterpret_cast<const float4 *>(q + (4 - ky) * p.pitch + 4);
                        const float v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const float4 w0 = *reinterpret_cast<const float4 *>(w + h * 40 + ky * 8);
                            const float wk[5] = {w0.x, w0.y, w0.z, w0.w, w[h * 40 + ky * 8 + 4]};
#pragma unroll
                            for (int kx = 0; kx < 5; ++kx)
#pragma unroll
                                for (int i = 0; i < 4; ++i) acc[h][i] = fmaf(v[i + 4 - kx], wk[kx], acc[h][i]);
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (c2 + h >= p.Cin) continue;
                    O *dst = static_cast<O *>(p.dX) + (static_cast<long long>(b) * p.Cin + c2 + h) * HW + y * Wd + x0;
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (x0 + i < Wd) store_value(dst + i, acc[h][i] * delta);
                }
            }
        }
        if (want_dw && rg < p.rg) {
            for (int y = rg; y < H; y += p.rg) {
                const float *xr = x_s + (ci_w * Hp + y + ky_w) * p.pitch;      // image row y + ky - 2
                const float *qr = qb + y * Wr * p.cop + q4 * 4;
                for (int x = 0; x < Wr; x += 4) {
                    const float4 a = *reinterpret_cast<const float4 *>(xr + x), c = *reinterpret_cast<const float4 *>(xr + x + 4);
                    const float v[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i) {                              // codes beyond the row's end are zero
                        const float4 q = *reinterpret_cast<const float4 *>(qr + (x + i) * p.cop);
#pragma unroll
                        for (int k = 0; k < 5; ++k) {
                            acc_w[0][k] = fmaf(q.x, v[i + k], acc_w[0][k]);
                            acc_w[1][k] = fmaf(q.y, v[i + k], acc_w[1][k]);
                            acc_w[2][k] = fmaf(q.z, v[i + k], acc_w[2][k]);
                            acc_w[3][k] = fmaf(q.w, v[i + k], acc_w[3][k]);
                        }
                    }
                }
            }
        }
    }
    if (!want_dw) return;
    // the row shares' sums -> one block of dW, which the copy engine adds to the others'
    __syncthreads();
    const int nout = p.Cout * p.Cin * 25;
    float *out_s = smem5, *part = smem5 + ((nout + 3) & ~3);         // [rg][cop][Cin][25]
    const int npart = p.cop * p.Cin * 25;
    if (rg < p.rg) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < 5; ++k) part[rg * npart + ((q4 * 4 + j) * p.Cin + ci_w) * 25 + ky_w * 5 + k] = acc_w[j][k];
    }
    __syncthreads();
    for (int i = tid; i < nout; i += kThreads5) {
        float s = 0.f;
        for (int r = 0; r < p.rg; ++r) s += part[r * npart + i];
        out_s[i] = s * delta;
    }
    tc::fence_async_proxy();
    __syncthreads();
    const int bulk = nout & ~3;                                      // whole 16-byte pieces; the rest by atomics
    if (tid == 0 && bulk > 0) {
        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;"
                     ::"l"(p.dW), "r"(tc::smem_u32(out_s)), "r"(bulk * 4) : "memory");
        tc::bulk_commit();
        tc::bulk_wait_read_all();
    }
    if (tid < nout - bulk) atomicAdd(p.dW + bulk + tid, out_s[bulk + tid]);
}

int floats5(const Direct5P &p) {
    const int Wr = p.pitch - 4, Hp = p.H + 4, cip = (p.Cin + 1) & ~1;
    const int tiles = (p.dX ? p.Cout * (p.plane + cip * 40) : 0) + (p.dW ? p.H * Wr * p.cop + p.Cin * Hp * p.pitch : 0);
    const int sums = p.dW ? ((p.Cout * p.Cin * 25 + 3) & ~3) + p.rg * p.cop * p.Cin * 25 : 0;
    return tiles > sums ? tiles : sums;
}

Direct5P plan5(const ConvShape &s, float *dW, void *dX) {
    Direct5P p{};
    p.dW = dW; p.dX = dX;
    p.B = static_cast<int>(s.B); p.Cin = static_cast<int>(s.Cin); p.Cout = static_cast<int>(s.Cout);
    p.H = static_cast<int>(s.H); p.Wd = static_cast<int>(s.W);
    p.pitch = (p.Wd + 3) / 4 * 4 + 4;
    p.cop = (p.Cout + 3) & ~3;
    p.co4 = p.cop / 4;
    p.rg = kThreads5 / (p.co4 * p.Cin * 5);
    if (p.rg > p.H) p.rg = p.H;
    p.plane = (p.H + 4) * p.pitch;
    if (p.plane % 8 == 0) {
        p.plane += 4;
        if (floats5(p) > kMaxFloats5) p.plane -= 4;                  // (fits as it is)
    }
    return p;
}

}  // namespace

// 5x5 layers whose weight gradient is one register tile per thread and whose image fits the shared memory.
bool direct5_supported(const ConvShape &s, bool want_dw, bool want_dx) {
    if (s.k != 5 || s.Cin > 64 || s.Cout > 256 || s.H > 256 || s.W > 256 || !(want_dw || want_dx)) return false;
    static float any;                              // only whether a product is wanted matters to the plan
    const Direct5P p = plan5(s, want_dw ? &any : nullptr, want_dx ? &any : nullptr);
    return p.co4 * p.Cin * 5 <= kThreads5 && floats5(p) <= kMaxFloats5;
}

// dW has been cleared.
int launch_direct5(dbp_ctx *ctx, const int8_t *codes, const void *X, const void *W, int io, const float *delta_p,
                   const ConvShape &s, float *dW, void *dX, bool dx_bf16) {
    Direct5P p = plan5(s, dW, dX);
    p.codes = codes; p.X = X; p.W = W; p.delta_p = delta_p;
    const int smem = floats5(p) * 4;
    // dW by itself with more images than SMs: two CTAs on an SM. A CTA that also makes dX is bound by its FMAs, which want the
    // registers of a whole SM; it keeps one to itself, for all of its images in turn. us by one, two: 1 -> 6 at 32x32, dW, batch 150:
    // 16.6, 15.2; 300: 21.5, 19.0; 600: 32.8, 27.3. 6 -> 16 at 16x16, both products, batch 150: 32.6, 34.9; 300: 45.3, 57.9; 600: 71.8, 72.2.
    const bool two = dX == nullptr && s.B > ctx->sm_count && floats5(p) <= kHalfFloats5;
    const long long cap = (two ? 2ll : 1ll) * ctx->sm_count;
    const unsigned grid = static_cast<unsigned>(s.B < cap ? s.B : cap);
    auto go = [&](auto kern) -> int {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxFloats5 * 4) != cudaSuccess)
            return fail_cuda("shared memory size");
        return cuda_ok(launch_chained(kern, dim3(grid), dim3(kThreads5), static_cast<size_t>(smem), ctx->stream, p));
    };
    if (two) return io == DBP_F32 ? go(direct5_kernel<float, float, 2>) : go(direct5_kernel<__nv_bfloat16, float, 2>);
    if (io == DBP_F32) return go(direct5_kernel<float, float, 1>);
    return dx_bf16 ? go(direct5_kernel<__nv_bfloat16, __nv_bfloat16, 1>) : go(direct5_kernel<__nv_bfloat16, float, 1>);
}

}  // namespace dbp
