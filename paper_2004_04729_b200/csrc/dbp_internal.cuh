// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "dbp.h"

namespace dbp {

constexpr int kSegment = DBP_SEGMENT;          // elements per sparse segment
constexpr int kWordsPerSegment = kSegment / 32;

// Device-side scalars of one context.
struct DeviceState {
    float delta;                        // step size of the internal quantization
    int nonfinite;                      // set when delta_z held NaN/Inf
    int tc_timeout;                     // a bounded wait of a tensor-core kernel expired
    unsigned long long nnz;             // non-zero codes of the internal quantization
    unsigned long long saturated;       // clipped codes since the last report
};

struct ProfSlot {
    cudaEvent_t begin, end;
    int kind;
};

struct Workspace {
    void *ptr = nullptr;
    size_t bytes = 0;
};

// A stride-2 layer's own tensors, while the tensor-core path runs it as a stride-1 layer on phase images.
struct StridedLayer {
    const void *X;                      // [B][Cin][H][W]
    void *dX;                           // the same shape, fp32 or the layer's type
    int dx_f32;
    float *dW;                          // [Cout][Cin][k][k]
    long long Cin;
    int H, W, phases;
};

// The gradient is routed from a pooled one by the statistics kernel, which writes it and adds it up in one pass: planes of
// 2h x 2w elements, w even.
struct PoolRouting {
    const float *g = nullptr;          // [planes][h][w]; null: the gradient is there
    const int8_t *argmax = nullptr;
    float *out = nullptr;
    int w = 0;
};

}  // namespace dbp

struct dbp_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    int sm_count = 148;
    dbp::DeviceState *state = nullptr;  // device
    double *partials = nullptr;         // device, statistics partial sums
    unsigned long long *wait_stats = nullptr;   // device, DBP_WAIT_SLOTS counters of SM clocks spent waiting
    int partial_blocks = 0;
    // The codes of a layer exist in two sets of buffers used in turn: with DBP_DW_ASYNC the dW kernels of
    // one call may still read their set while the next call's quantization writes the other one.
    dbp::Workspace dense_codes[2];      // int8 per element of delta
    dbp::Workspace x_padded[2];         // activations re-written as 16-byte aligned bf16 planes, one per set of codes
    dbp::Workspace db_sums;             // bias gradient: counters that are zero between calls, then partial sums
    dbp::Workspace rows_x, rows_w;      // operands re-written as bf16 rows the copy engine can address: a linear layer's X, W
    dbp::Workspace codes16[2];          // bf16 code planes for the TMA-fed kernels
    dbp::Workspace w_taps;              // fp32 weights as [Cout][k*k][Cin]
    dbp::Workspace codes_nhwc[2];       // bf16 codes [B][position][Cout] for the TMA-fed 3x3 kernels
    dbp::PoolRouting pooled;            // set while dithered_conv_backward_pooled runs a call whose statistics kernel routes the gradient
    const uint8_t *next_mask = nullptr; // ReLU mask for the next backward call (dbp_set_relu_mask)
    dbp::Workspace dz_tmp;              // delta_z = delta_a (.) mask when that call cannot fold the mask into its loads
    dbp::Workspace codes_stack[2];      // the same codes with G images stacked into one tall image (tiny planes, dW)
    const void *phase_w_src = nullptr;  // that layer's own weights: its W argument is a workspace for the phase weights, not yet written
    float *phase_dw_out = nullptr;      // that layer's dW: the 3x3 weight-gradient kernels write it directly when they run in phase mode ...
    bool phase_dw_done = false;         // ... and say so here
    int phase_cin = 0;                  // > 0 while a stride-2 3x3 layer runs as a stride-1 layer on phase images: its own channel count
    const dbp::StridedLayer *strided = nullptr;   // set while a stride-2 layer runs as a stride-1 layer on phase images made inside
    dbp::Workspace s2_x, s2_w, s2_dx, s2_dw;   // stride-2 layers: phase images of X, phase weights, and the two products in that layout
    float *delta_sets = nullptr;        // device float[2]: the step size that belongs to each set
    int code_set = 0;                   // the set the next call writes
    cudaEvent_t ev_set_free[2] = {nullptr, nullptr};   // recorded on the dW stream after the set's last reader
    bool set_busy[2] = {false, false};
    bool aux_pending = false;           // dW work on the second stream that the caller's stream is not yet ordered after
    dbp::Workspace dw_acc;              // fp32 [tap][Cout][Cin] that the 3x3 dW CTAs add into; zero between calls
    bool dw_acc_clean = false;
    dbp::Workspace io[8];               // staging for the *_host entry points
    // *_host entry points: X goes up and dX comes down on streams of their own, so that the two
    // directions of the host link work at the same time; the events order them against the
    // kernels (dX done -> its read-back may start; X up -> the dW kernels may start)
    // the dense dW kernels of a layer run beside its dX kernel on a stream of their own (they only
    // share inputs): forked after the quantization, joined before the call returns to the caller's stream
    cudaStream_t aux = nullptr;
    cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    cudaEvent_t ev_x_up = nullptr, ev_dx_done = nullptr;
    cudaEvent_t hook_after_dx = nullptr, hook_before_dw = nullptr;   // set only during a *_host call
    // density above which the dense path is preferred. Measured (sparse against dense time for a 1x1, a 3x3 and a
    // linear layer, densities 22 % ... 0.6 %): the tensor-core path is 6.6x to 14x faster at every density, the gather
    // kernels' time being mostly the scan of the dense codes; so wherever the dense path exists it is the default.
    float crossover = 0.0f;
    // densities measured so far, by layer shape (the path choice of a call uses its own shape's entry)
    struct DensityEntry { unsigned long long key; float density; };
    std::vector<DensityEntry> densities;
    unsigned long long nnz_host_key = 0;         // shape whose read-back is in flight
    unsigned long long *nnz_host = nullptr;   // pinned: asynchronous read-back of nnz
    long long nnz_host_numel = 0;
    cudaEvent_t nnz_event = nullptr;
    bool nnz_pending = false;
    bool profiling = false;
    unsigned prof_mask = 0xffffffffu;   // kinds that are timed while profiling is on
    std::vector<dbp::ProfSlot> prof;    // event pairs, reused after every read
    size_t prof_used = 0;
    double prof_ms[DBP_K_COUNT] = {0};
    long long prof_launches[DBP_K_COUNT] = {0};
};

namespace dbp {

int ws_reserve(dbp_ctx *ctx, Workspace &w, size_t bytes);

// Where a quantizer takes the step size from: the statistics kernel's partial sums, or a device scalar.
struct StepSource {
    const float *given = nullptr;
    const double *partials = nullptr;   // (sum, sum of squares) of each statistics block, about the pivot
    int nparts = 0;
    double inv_numel = 0;
    float scale = 0.f;
    int late = 0;                       // the statistics kernel writes the gradient: it is read behind the wait for that kernel
    float *publish[3] = {nullptr, nullptr, nullptr};   // where the quantizer writes it for the kernels behind it
};

// ---- nsd_kernels.cu
// Work the statistics kernel does on the side for the layer's product kernels (its blocks have time to spare
// and this saves launches): clearing a buffer (16-byte aligned, a multiple of 16 bytes), and re-laying 3x3
// weights [Cout][Cin][9] as [taps][Cout][Cin rounded up to 8] bf16 (taps = 9 for bf16 weights; 18 for fp32 weights, split into
// two bf16 pieces: taps 0-8 the rounded values, 9-17 what the rounding left over).
// Rows of a matrix as bf16 rows of `pitch` values (a multiple of 8, extra columns zero), which the copy engine can
// address: fp32 rows become two pieces, rows * pitch apart (the rounded values, and the remainders rounded).
struct RowsJob {
    const void *src = nullptr;
    void *dst = nullptr;
    int f32 = 0;
    long long rows = 0, cols = 0, pitch = 0;
};
struct SideJobs {
    PoolRouting pool;                  // (the only jobs beside it: clearing a buffer)
    RowsJob rows[2];
    int nrows = 0;
    void *zero = nullptr;
    size_t zero_bytes = 0;             // a multiple of 4
    const void *w_src = nullptr;       // null: no weights to re-lay
    void *w_dst = nullptr;
    int w_f32 = 0;
    long long Cout = 0, Cin = 0;
    int phase_cin = 0;                 // > 0: w_src holds a stride-2 layer's own weights [Cout][phase_cin][9], Cin = 4 phase_cin
    int skip_dead = 0;                 // ... whose taps that are zero by construction nobody reads: they are not written
};
// publish: where the quantizer is to write the step size beside the context's state (entries may be null); *step tells
// the quantizer where to take it from
int launch_statistics(dbp_ctx *ctx, const void *delta, int dtype, long long numel, float scale,
                      const float *delta_in, float *const (&publish)[2], unsigned long long *nnz_out, StepSource *step,
                      const SideJobs &jobs = SideJobs(), const uint8_t *mask = nullptr);
// beside: the kernel before it on the stream is the quantizer; the job runs beside it
int launch_rows_job(dbp_ctx *ctx, const RowsJob &job, bool beside);
int launch_quantize(dbp_ctx *ctx, const void *delta, int dtype, long long numel,
                    unsigned long long seed, const StepSource &step, uint32_t *bitmap,
                    uint16_t *offsets, int8_t *values, int8_t *dense,
                    unsigned long long *nnz_out);
// ---- nsd_dense.cu: the same codes, dense array only (no sparse structure)
// either dense: int8 codes in delta's order, or planes_bf16: bf16 codes as [numel / hw][pitch], pitch a multiple of 8
int launch_quantize_dense(dbp_ctx *ctx, const void *delta, int dtype, long long numel,
                          unsigned long long seed, const StepSource &step, int8_t *dense,
                          void *planes_bf16, long long hw, long long pitch, bool count, const uint8_t *mask = nullptr);
// position-major bf16 codes [B][HW][C] for the TMA-fed 3x3 kernels
int launch_quantize_nhwc(dbp_ctx *ctx, const void *delta, int dtype, long long B, long long C, long long HW,
                         unsigned long long seed, const StepSource &step, void *codes_nhwc, bool count,
                         void *codes_stack = nullptr, int plane_w = 0, const uint8_t *mask = nullptr);
int launch_decode(dbp_ctx *ctx, const uint32_t *bitmap, const uint16_t *offsets,
                  const int8_t *values, long long numel, int8_t *dense);

// ---- small_linear.cu: the whole backward pass of a small fp32 linear layer in two chained launches
bool small_linear_fits(const dbp_ctx *ctx, long long B, long long N, long long K, bool want_dw, bool want_dx);
int launch_small_linear(dbp_ctx *ctx, const float *delta, const float *X, const float *W, long long B, long long N,
                        long long K, unsigned long long seed, float scale, const float *delta_in, float *dW, float *dX,
                        float *db, float *delta_set, const uint8_t *mask = nullptr);

// ---- linear_tc.cu: both products of a linear layer in one launch; codes as bf16 [B][linear_pitch(N)]
struct LinearPlan {
    int TN = 0;                       // columns per tile
    int MA = 1;                       // accumulators (of 128 rows) per tile
    long long dw_split = 1, dw_per_split = 0;   // > 1: dW is added up from parts and must have been cleared
};
bool linear_tc_supported(long long B, long long N, long long K);
long long linear_pitch(long long cols);
LinearPlan linear_plan(const dbp_ctx *ctx, long long B, long long N, long long K, int pieces, bool want_dw, bool want_dx);
// X, W: bf16 [pieces][rows][pitch]; pieces = 2 for fp32 operands split by a RowsJob
int launch_linear_products(dbp_ctx *ctx, const LinearPlan &pl, const void *codes, const void *X, const void *W, int pieces,
                           long long x_pitch, long long w_pitch, const float *delta_p, long long B, long long N, long long K,
                           float *dW, void *dX, bool dx_bf16, int *err_flag);

// ---- bias_grad.cu: db from bf16 codes, rows [rows][cols rounded up to 8] or planes [B][channels][pitch]
// beside: the call may run beside the kernel before it on the stream (a product, which writes nothing it reads)
int launch_column_sums(dbp_ctx *ctx, const void *codes, long long rows, long long cols, const float *delta_p, float *db,
                       bool beside);
int launch_plane_sums(dbp_ctx *ctx, const void *codes, long long B, long long channels, long long hw, long long pitch,
                      const float *delta_p, float *db, bool beside);

// ---- product_kernels.cu
struct ConvShape {
    long long B, Cin, Cout, H, W;
    int k;
};
// weights as [Cout][k*k][Cin]; kept in their own dtype unless to_f32
int launch_weight_taps(dbp_ctx *ctx, const void *W, int dtype, const ConvShape &s, void *w_taps,
                       bool to_f32);
int launch_conv_dx_streamed(dbp_ctx *ctx, const int8_t *codes, const void *w_taps, int w_dtype,
                            const float *delta_p, const ConvShape &s, void *dX, bool dx_bf16);
int launch_conv_dx(dbp_ctx *ctx, const int8_t *codes, const float *w_taps, const float *delta_p,
                   const ConvShape &s, void *dX, bool dx_bf16);
int launch_conv_dw(dbp_ctx *ctx, const int8_t *codes, const void *X, int dtype,
                   const float *delta_p, const ConvShape &s, float *dW);
int launch_conv_dw_streamed(dbp_ctx *ctx, const int8_t *codes, const void *X, int dtype,
                            const float *delta_p, const ConvShape &s, float *dW);
// ---- tma_dx.cu: 1x1 dX with TMA-fed operands; codes as bf16 planes [B*Cout][tma_code_pitch]
bool tma_dx_supported(const ConvShape &s, int io);
long long tma_code_pitch(const ConvShape &s);
// W: bf16 [pieces][Cout][w_pitch]; X: bf16 [pieces of B images][Cin][x_pitch] (pitches multiples of 8)
int launch_tma_dx(dbp_ctx *ctx, const void *codes_bf16, const void *W, int pieces, long long w_pitch, const float *delta_p,
                  const ConvShape &s, void *dX, bool dx_bf16, int *err_flag);
// ---- tma_dw.cu: 1x1 dW with TMA-fed operands (same code planes)
int launch_tma_dw(dbp_ctx *ctx, const void *codes_bf16, const void *X, int pieces, long long x_pitch, const float *delta_p,
                  const ConvShape &s, float *dW, int *err_flag);
// ---- tc3_tma_dx.cu / tc3_tma_dw.cu: 3x3 products with TMA-fed operands; codes as bf16 [B][H*W][Cout rounded up to 8]
// dx_f32: an fp32 dX is wanted, to the accuracy of every other
bool tc3_tma_supported(const ConvShape &s, int io, bool dx_f32);
// io: the operands' type; fp32 weights / activations are split into two bf16 pieces on the way in
// weights_ready: ctx->w_taps already holds the re-laid weights (the statistics kernel did it on the side)
// lean (may be null): the kernel may confine itself to half of every SM, so that the dW kernel (half) runs beside it; set to
// whether it did. dX is the same either way.
int launch_tc3_tma_dx(dbp_ctx *ctx, const void *codes_nhwc, const void *W, int io, const float *delta_p,
                      const ConvShape &s, void *dX, bool dx_bf16, int *err_flag, bool weights_ready = false, bool *lean = nullptr);
// ---- tc3_rows_dx.cu: the same for small planes, a row of several images at a time
struct RowsPlan {
    int nimg = 0, KS = 1;               // images per tile, CTAs that share its reduction
};
// max_cols: accumulator columns of a tile, at most; lean: as for launch_tc3_tma_dx
double tc3_rows_plan(const dbp_ctx *ctx, const ConvShape &s, int pieces, int max_cols, RowsPlan *plan);
int launch_tc3_rows_dx(dbp_ctx *ctx, const RowsPlan &plan, const void *codes_nhwc, int pieces, const float *delta_p, const ConvShape &s,
                       void *dX, bool dx_bf16, int *err_flag, bool *lean);
constexpr int kRowsLeanCols = 128, kRowsMaxCols = 256;       // accumulator columns of a tile: that fits half an SM, at most
// Dynamic shared memory of a kernel two of whose CTAs share an SM (228 KB, of which a CTA takes 1 KB and the 1 KB of its own variables)
constexpr size_t kHalfSm = 112 * 1024;
// X: bf16 planes of x_pitch values, pieces of every image one after the other
int launch_tc3_tma_dw(dbp_ctx *ctx, const void *codes_nhwc, const void *X, int pieces, long long x_pitch, const float *delta_p,
                      const ConvShape &s, float *dW, int *err_flag, bool half, bool overlapped);
bool tc3_dw_fits_half(const ConvShape &s);
// fp32 activations split and stacked for it (out: [2][B / G][Cin][pitch]); beside: as for launch_rows_job
int launch_x_stacked(dbp_ctx *ctx, const float *X, void *out, const ConvShape &s, int stack_g, bool beside);
// Planes of fewer than 64 positions: how many images of a batch to stack into one tall image (one zero row after
// every image) for the weight-gradient kernel, whose work comes in segments of one image; 0: do not stack.
int tc3_stack_images(const ConvShape &s, int io);
int launch_bias_grad(dbp_ctx *ctx, const int8_t *codes, const float *delta_p, const ConvShape &s,
                     float *db);
int launch_relu_backward(dbp_ctx *ctx, const float *da, const uint8_t *mask, float *dz,
                         long long n);
int launch_maxpool_backward(dbp_ctx *ctx, const float *g, const int8_t *argmax, float *out,
                            long long planes, long long h, long long w);

// ---- fused1x1.cu: quantization and both products of a thin bf16 1x1 layer in one kernel (dW cleared by the caller, bf16 dX)
bool fused1x1_supported(const dbp_ctx *ctx, const ConvShape &s, int io);
int launch_fused1x1(dbp_ctx *ctx, const void *delta, const void *X, const void *W, const ConvShape &s, unsigned long long seed,
                    const StepSource &step, float *dW, void *dX, int *err_flag);

// ---- direct5.cu: both products of a 5x5 layer of few channels by FMAs on the dense codes (dW cleared by the caller)
bool direct5_supported(const ConvShape &s, bool want_dw, bool want_dx);
int launch_direct5(dbp_ctx *ctx, const int8_t *codes, const void *X, const void *W, int io, const float *delta_p,
                   const ConvShape &s, float *dW, void *dX, bool dx_bf16);

// ---- strided_conv.cu: layout changes around a stride-2 layer run as a stride-1 layer on the input's phase images
// (phases = 4: all four, channel (py*2+px)*Cin + ci; phases = 1: the even rows and columns only)
int launch_phases_of(dbp_ctx *ctx, const void *X, void *Xp, int io, long long B, long long Cin, int H, int W, int phases);
// the same as bf16 rows for the copy engine (fp32: two pieces), [pieces][B][phases * Cin][pitch]; beside: as launch_rows_job
int launch_phase_rows(dbp_ctx *ctx, const void *X, void *Xp, int io, long long B, long long Cin, int H, int W, int phases,
                      long long pitch, bool beside);
int launch_from_phases(dbp_ctx *ctx, const void *dXp, void *dX, int f32, long long B, long long Cin, int H, int W, int phases);
int launch_phase_weights(dbp_ctx *ctx, const void *W, void *Wp, int io, long long Cout, long long Cin);
int launch_strided_dw(dbp_ctx *ctx, const float *dWp, float *dW, long long Cout, long long Cin);

// ---- selftest.cu
int launch_bounded_wait_selftest(dbp_ctx *ctx, long long budget);
// fp32 FMA throughput of the device (dependent chains on every lane of every SM), TFLOP/s
int measure_fma_peak(dbp_ctx *ctx, double *tflops);

// Brackets one kernel launch with events while profiling is on.
struct KernelTimer {
    dbp_ctx *ctx;
    ProfSlot *slot = nullptr;
    KernelTimer(dbp_ctx *c, int kind) : ctx(c) {
        if (!c->profiling || !((c->prof_mask >> kind) & 1u)) return;
        if (c->prof_used == c->prof.size()) {
            ProfSlot s;
            if (cudaEventCreate(&s.begin) != cudaSuccess) return;
            if (cudaEventCreate(&s.end) != cudaSuccess) { cudaEventDestroy(s.begin); return; }
            s.kind = kind;
            c->prof.push_back(s);
        }
        slot = &c->prof[c->prof_used++];
        slot->kind = kind;
        cudaEventRecord(slot->begin, c->stream);
    }
    ~KernelTimer() {
        if (slot) cudaEventRecord(slot->end, ctx->stream);
    }
};

// An accumulator of the tensor cores is truncated, not rounded, when an MMA adds to it: a sum of terms of one sign comes out
// low by up to 1.7e-8 of itself per MMA (measured: bf16 1x1 dW, 680 and 1360 MMAs: 0.9e-5 and 2.3e-5; fp32 3x3 dW, 2100
// MMAs: 4.8e-5). Longer reductions are cut into parts of at most this many, which are added with rounding: at most 0.9e-5.
// (fp32 operands enter as two bf16 pieces, whose sum is within 2^-17 of the value: errors of either sign, which average out
// over the terms unless all operands have the same mantissa.)
constexpr int kMaxMmas = 512;

// Split of a K loop of `kunits` steps over CTAs when `tiles` output tiles exist and one CTA fits
// per SM: the CTAs run in ceil(tiles * split / sms) waves of ceil(kunits / split) steps each, so
// a split that spills a few CTAs into another wave doubles the time. Picks the split with the
// fewest wave-steps (a CTA's fixed cost counted as two steps, a small charge per split for the
// partial sums) among those of at most max_per steps per CTA; *per_split receives the steps per CTA.
// The returned split has no empty part.
inline long long choose_split(long long tiles, long long kunits, int sms, long long max_per, long long *per_split) {
    const long long least = (kunits + max_per - 1) / max_per;
    long long best = least, best_per = max_per;
    double best_cost = 1e300;
    long long smax = kunits < 4ll * sms ? kunits : 4ll * sms;
    if (smax < least) smax = least;
    for (long long want = least; want <= smax; ++want) {
        const long long per = (kunits + want - 1) / want, split = (kunits + per - 1) / per;
        const long long waves = (tiles * split + sms - 1) / sms;
        const double cost = static_cast<double>(waves) * static_cast<double>(per + 2) + 0.05 * static_cast<double>(split);
        if (cost < best_cost) { best_cost = cost; best = split; best_per = per; }
    }
    *per_split = best_per;
    return best;
}

// Records where a CUDA call failed and what the runtime said (read back with dbp_last_error);
// returns DBP_ECUDA.
int fail_cuda(const char *what, cudaError_t e);
inline int fail_cuda(const char *what) { return fail_cuda(what, cudaGetLastError()); }

// Every kernel launch of the library passes here (a process-wide count, read by dbp_kernel_launches).
void note_launch();

inline int cuda_ok(cudaError_t e) { return e == cudaSuccess ? DBP_OK : fail_cuda("launch", e); }

// Programmatic dependent launch: a kernel launched with launch_chained may become resident while
// the kernel before it in the stream is still draining; it must call chain_wait() before it
// touches global memory (the wait returns once the earlier kernel has completed and its writes
// are visible), and chain_release() lets the kernel after it do the same. Both are no-ops for a
// kernel launched the ordinary way.
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                  Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
// The same for a grid of clusters of `cluster` consecutive blocks.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained_cluster(void (*kern)(KArgs...), unsigned ctas, unsigned cluster, dim3 block, size_t smem,
                                          cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    note_launch();
    return cudaLaunchKernelEx(&cfg, kern, static_cast<KArgs>(args)...);
}
// Dynamic shared memory that a kernel may be launched with. The limit belongs to the function on the device and not to a launch, and
// threads with a context each set it at the same time: every call sets one value, the most that any launch of the kernel asks for.
constexpr int kMostShared = 226 * 1024;          // a CTA has 227 KB, 1 KB of them for its own variables
template <typename Kern>
inline cudaError_t allow_shared(Kern kern, int most = kMostShared) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}
#endif

}  // namespace dbp
