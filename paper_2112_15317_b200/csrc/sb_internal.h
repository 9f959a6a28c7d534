// Internal declarations shared by the host-side planner (sb_api.cu) and the kernel files.
// Nothing here is part of the public C ABI (see include/splitbrain.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>

#include <cstdlib>
#include <utility>

namespace sb {

constexpr int MAX_PARTS = 64;  // upper bound on R and K

// ---------------------------------------------------------------------------------------------
// Programmatic dependent launch.  Every kernel of the library starts with pdl_prologue(): it waits until the
// kernels it depends on have completed (griddepcontrol.wait, a no-op for a normally launched kernel) and
// then lets the next kernel in the stream start launching (griddepcontrol.launch_dependents), so that the
// next kernel's launch latency and set-up overlap this kernel's execution.  Nothing is read from or written
// to global memory before the wait.  SB_PDL=0 in the environment launches everything the classic way.
// ---------------------------------------------------------------------------------------------
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_prologue() { pdl_wait(); pdl_trigger(); }
#endif
// Tuning constants of the planner.  The shipped library uses the compiled-in defaults; a development build
// (-DSB_DEV_TUNING) lets an environment variable of the same name override each one for A/B measurements.
inline double tune(const char* name, double dflt)
{
#ifdef SB_DEV_TUNING
    const char* e = getenv(name);
    return e ? atof(e) : dflt;
#else
    (void)name;
    return dflt;
#endif
}
// (the calling thread can switch the attribute off for the launches it enqueues next: pdl_classic() = 1 ... = 0)
inline int& pdl_classic() { static thread_local int off = 0; return off; }
// Set by the calling thread around a launch whose predecessor in the stream is known not to have written the layer's weights
// (a kernel of the same forward or backward pass): the tensor-core kernel may then fetch weights before it waits for it.
inline int& weights_first() { static thread_local int on = 0; return on; }
inline bool pdl_enabled()
{
    static const bool on = [] { const char* e = getenv("SB_PDL"); return !(e && e[0] == '0'); }();
    return on && !pdl_classic();
}
// Scheduling priority of the calling thread's next launches (0 = least, negative before it): which of the kernels that are ready gets
// the SMs another one's finished blocks leave.  In a graph it counts where the graph is instantiated with its nodes' priorities.
inline int& launch_priority() { static thread_local int p = 0; return p; }
template <typename... KArgs, typename... Args>
inline cudaError_t pdl_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    int n = 0;
    if (pdl_enabled()) {
        at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (launch_priority() != 0) {
        at[n].id = cudaLaunchAttributePriority;
        at[n++].val.priority = launch_priority();
    }
    cfg.attrs = at;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kern, KArgs(std::forward<Args>(args))...);
}
// Raises a kernel's dynamic shared-memory limit, once per device (the attribute belongs to the device's copy of the function).
template <auto Kernel>
inline cudaError_t raise_smem_limit(int bytes)
{
    static bool done[64] = {false};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (done[dev]) return cudaSuccess;
    e = cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    done[dev] = e == cudaSuccess;
    return e;
}
#define SB_LAUNCH(kern, grid, block, smem, st, ...) (void)::sb::pdl_launch((kern), dim3(grid), dim3(block), (size_t)(smem), (st), __VA_ARGS__)


// Pointer table for per-replica caller buffers (inputs, labels): passed by value to kernels.
struct PtrTab {
    const void* p[MAX_PARTS];
};

// Learning rate and momentum of an update: by value, or read from two device words (dev != nullptr).  A captured iteration carries
// values as long as they stay the same; once they have changed it is captured with the device words, so that a learning-rate
// schedule costs one 1-block kernel per change instead of a capture and an instantiation (2.2 ms at VGG-16 size; values in
// every kernel: VGG-16 at 32x32, batch 128, 0.5 % faster than the words).
struct Hyper {
    float lr, mu;
    const float* dev;
#ifdef __CUDACC__
    __device__ __forceinline__ float rate() const { return dev ? __ldg(dev) : lr; }
    __device__ __forceinline__ float decay() const { return dev ? __ldg(dev + 1) : mu; }
#endif
};

// Device status word codes (written by kernels that give up on a bounded wait).
enum : uint32_t { DEV_OK = 0, DEV_TIMEOUT_TMA = 1, DEV_TIMEOUT_MMA = 2, DEV_TIMEOUT_EPI = 3, DEV_PAIR_TMEM = 4 };

// ---------------------------------------------------------------------------------------------
// CUDA-core ("SIMT") kernels: the float mode, odd channel counts, and the cross-check path.
// All launchers return the cudaError_t of the launch.  `bf16` selects the activation dtype
// (false: float, true: __nv_bfloat16) of every T-typed pointer.
// ---------------------------------------------------------------------------------------------

struct ConvSimtArgs {
    const void* in;       // [B,H,W,Cin] activation dtype (ignored when tab != nullptr)
    const PtrTab* tab;    // optional: R per-replica input pointers (host pointer to the table)
    int b_per_rep;
    const void* w;        // [Cout,3,3,Cin] activation dtype (float master or bf16 shadow)
    const float* bias;    // [Cout]
    void* out;            // [B,H,W,Cout] activation dtype
    int B, H, W, Cin, Cout;
    int relu;
};
struct WgradSimtArgs {
    const void* x;        // [B,H,W,Cin] (ignored when tab != nullptr)
    const PtrTab* tab;
    int b_per_rep;
    const void* dy;       // [B,H,W,Cout]
    float* part;          // partial sums
    int B, H, W, Cin, Cout;
};

// 3x3 convolution (taps = 9) or fully-connected layer (taps = 1, H = W = 1) on CUDA cores (sb_contract_simt.cu) or, for float
// operands, on tensor cores with every float as three bf16 terms (sb_contract_umma.cu).
enum { CMODE_FWD = 0, CMODE_DGRAD = 1, CMODE_WGRAD = 2 };
struct ContractPlan { int bm = 64, bn = 64, iters = 0, splits = 1; bool umma = false; };     // block tile, reduction steps (16 or, umma, 64) per split, splits
// max_part_floats: room for split partial sums ([splits][result], for WGRAD with the bias gradient behind each)
// umma: the tensor-core form may be chosen (float operands; the layer input is one buffer)
ContractPlan contract_plan(int mode, int B, int H, int W, int taps, int Cin, int Cout, size_t max_part_floats, bool umma);
struct ContractArgs {
    int mode, taps, B, H, W, Cin, Cout;
    const void *act, *wt, *dy;             // layer input (or tab), weights [Cout][taps][Cin], output gradient, in the activation dtype
    const PtrTab* tab; int tab_imgs;       // optional: the layer input as per-replica buffers of tab_imgs images
    ContractPlan plan;
    float* part; long split_stride;        // splits > 1: partial sums.  WGRAD: always where the gradient (or its splits) goes,
    long bias_off;                         // and the bias gradient's place relative to it
    void* out; float* out32;               // FWD / DGRAD result (out32: float instead of the activation dtype)
    const float* bias; int relu;           // FWD
    const void* ref;                       // DGRAD: zero where ref <= 0
    uint32_t* status;                      // device status word of the bounded waits
    const __nv_bfloat16* wterms;           // umma, FWD / DGRAD: the weights as three planes of bf16 terms, wterms_stride elements apart (or nullptr)
    size_t wterms_stride;
};
cudaError_t launch_contract(const ContractArgs& a, bool bf16, cudaStream_t st);
bool contract_umma_ok(int taps, int Cin, int Cout);
bool contract_umma_whole_taps(int mode, int Cin, int Cout);      // a reduction chunk never crosses taps: the forms that fetch by TMA
cudaError_t launch_split_weights(const float* w, __nv_bfloat16* terms, size_t n, size_t stride, cudaStream_t st);     // n, stride: multiples of 4
cudaError_t launch_contract_umma(const ContractArgs& a, cudaStream_t st);      // (without the second kernel of a split FWD / DGRAD)

// Input-layer convolution (Cin of 1, 3 or 4; Cout a multiple of 8): dedicated forward and weight+bias
// gradient kernels.  The gradient kernel writes conv_in_wgrad_blocks() partial buffers of
// Cout*9*Cin + Cout floats each (weights, then bias) into a.part, to be reduced in block order.
bool conv_in_supported(int Cin, int Cout);
cudaError_t launch_conv_in_fwd(const ConvSimtArgs& a, bool bf16, cudaStream_t st);
int conv_in_wgrad_blocks(int B, int H, int W);
cudaError_t launch_conv_in_wgrad(const WgradSimtArgs& a, bool bf16, cudaStream_t st);

struct XentArgs;
// Narrow FC layer (out <= 16): pass 0 forward, 1 weight+bias gradient, 2 input gradient.
struct FcNarrowArgs {
    int pass;
    const void* X; const PtrTab* tab; int tab_b;   // [B,in] activations (or R per-replica buffers of tab_b rows)
    const void* W;                                 // [out,in] activation dtype
    const float* bias; void* Y; float* Y32; int relu;   // forward outputs (either may be null)
    const void* dY; float* dW; float* db;          // gradient inputs/outputs
    const void* ref; void* dX;                     // dgrad: optional ReLU mask source and output [B,in]
    int B, in_f, out_f;
    const XentArgs* xent;                          // forward of the logits layer: the loss layer's row losses and dZ in the same kernel
                                                   // (launch_softmax_xent's bits; the mean loss is left to launch_loss_mean)
};
bool fc_narrow_supported(int out_f, int B);
cudaError_t launch_fc_narrow(const FcNarrowArgs& a, bool bf16, cudaStream_t st);

// part[s][n] = sum over the rows of split s of in[row][n] (bf16, N a multiple of 8).
cudaError_t launch_colsum(const void* in, float* part, int M, int N, int splits, cudaStream_t st);
// Elements from `at` on lie `by` further on where a reduce writes (or updates) them: a layer's bias vector behind the padding of its weights.
struct Gap {
    size_t at = 0, by = 0;
    __host__ __device__ size_t over(size_t i) const { return i < at ? i : i + by; }
    bool by4() const { return at % 4 == 0 && by % 4 == 0; }
};
// out[i] = sum_{s<splits} part[s*stride + i], s ascending.
cudaError_t launch_reduce_partials(const float* part, size_t stride, float* out, size_t n, int splits, cudaStream_t st, Gap gap = Gap{});
// the same ordered sum, consumed at once by the SGD step of the n parameters at w / v (shadow: their bf16 copies or nullptr)
cudaError_t launch_reduce_sgd(const float* part, size_t stride, size_t n, int splits, float* w, float* v, __nv_bfloat16* shadow,
                              Hyper hy, cudaStream_t st, Gap gap = Gap{});

struct PoolArgs {
    const void* x;  // [B,H,W,C]
    void* p;        // [B,H/2,W/2,C]
    uint8_t* idx;   // [B,H/2,W/2,C]
    int B, H, W, C;
};
cudaError_t launch_pool_fwd(const PoolArgs& a, bool bf16, cudaStream_t st);
struct PoolBwdArgs {
    const void* dp;      // [B,H/2,W/2,C] gradient w.r.t. the pooled output
    const uint8_t* idx;
    const void* p;       // pooled output (ReLU mask source) or nullptr for no mask
    void* dx;            // [B,H,W,C]
    int B, H, W, C;
};
cudaError_t launch_pool_bwd(const PoolBwdArgs& a, bool bf16, cudaStream_t st);

struct XentArgs {
    const float* logits;  // [B,C]
    PtrTab labels;        // R pointers to int32 [b]
    int b_per_rep;
    float* row_loss;      // [B]
    float* loss;          // [1] mean over rows
    void* dZ;             // [B,C] activation dtype: (softmax - onehot)/B
    unsigned int* counter; // zero-initialised word; left at zero
    int B, C;
    // Sub-batch use (modulo schedule): the rows above are a slice of a larger batch.  scale_B > 0 replaces B in the
    // 1/B of dZ; loss_rows > 0 makes the mean loss the sum of loss_base[0 .. loss_rows) divided by loss_rows.
    int scale_B = 0;
    const float* loss_base = nullptr;
    int loss_rows = 0;
};
cudaError_t launch_softmax_xent(const XentArgs& a, bool bf16, cudaStream_t st);
cudaError_t launch_loss_mean(const XentArgs& a, cudaStream_t st);

// Modulo layer as an explicit copy (sub-iteration schedule): R replicas of b rows, K slices of b/K rows each.
// gather : dst[k*(R*b/K) + r*(b/K) + i] = src[r*b + k*(b/K) + i]   (rows of `row_bytes` bytes, a multiple of 16)
// scatter: the inverse.  labels (optional, gather only): int32 per row, read through the per-replica table.
struct ModuloCopyArgs {
    const void* src;
    void* dst;
    size_t row_bytes;
    int R, b, K;
    int scatter;               // 0: gather, 1: scatter
    const PtrTab* labels;      // gather only: R pointers to int32 [b]; nullptr = no labels
    int32_t* labels_out;       // [R*b] in sub-iteration order
};
cudaError_t launch_modulo_copy(const ModuloCopyArgs& a, cudaStream_t st);

// Dropout layer on a [rows, width] activation matrix (units = drop probability * 65536): y = keep ? x / (1 - p) : 0 with the
// keep bit of logical element (row, column) drawn by a counter-based generator from `state` = {seed lo, seed hi, iteration}
// (device memory) and the layer index; backward: dx = dy / (1 - p) (dy arrives zero where the output was zero).
// sub_bk > 0: the rows are sub-iteration sub_k of the modulo schedule (sub_bk rows of each replica's sub_b); masks follow the batch rows
cudaError_t launch_dropout_fwd(const void* x, void* y, size_t rows, int width, const uint32_t* state, int layer, int units, bool bf16, cudaStream_t st,
                               int sub_bk = 0, int sub_b = 0, int sub_k = 0);
cudaError_t launch_dropout_bwd(const void* dy, void* dx, size_t n, int units, bool bf16, cudaStream_t st);
// mode 0: state <- {seed, iteration}; mode 1: iteration += 1
cudaError_t launch_dropout_state(uint32_t* state, int mode, uint64_t seed, uint32_t iteration, cudaStream_t st);

cudaError_t launch_sgd(float* w, float* v, const float* g, __nv_bfloat16* shadow, size_t n, Hyper hy, cudaStream_t st);
// writes {lr, mu} to the two words a Hyper with `dev` set reads
cudaError_t launch_hyper(float* dev, float lr, float mu, cudaStream_t st);
// copies the loss and the status word behind it to pinned host memory (a memcpy node started 4 to 9 us after the last kernel)
cudaError_t launch_report(const float* words, uint32_t* host, cudaStream_t st);
cudaError_t launch_to_bf16(const float* w, __nv_bfloat16* shadow, size_t n, cudaStream_t st);

enum { EPI_BIAS_ACT = 0, EPI_MASK = 1 };
// Ordered sum of split-reduction partial sums [split][rows][N] followed by the GEMM epilogue
// (epi = EPI_BIAS_ACT or EPI_MASK below).
struct SplitKEpiArgs {
    const float* part; size_t split_stride; int splits;
    long rows; int N;
    int epi; const float* bias; int relu; const void* ref;
    void* out; int out_f32;
};
cudaError_t launch_splitk_epilogue(const SplitKEpiArgs& a, bool bf16, cudaStream_t st);

// Pooling next to a contraction, offered by the calling thread around its launch: where the reduction is split, the epilogue kernel of the
// split sums does it in the same pass and sets `done`; elsewhere the offer is left untouched.  H, W, C are the pool layer's input.
//   forward (dx == nullptr): the result is that input; p and idx are the pool layer's output
//   backward: the result is the gradient of the pool layer's output; idx and mask (its output, or nullptr) lead it on to dx
struct SplitPool { int H, W, C; void* p; uint8_t* idx; const void* mask; void* dx; bool done; };
inline SplitPool*& split_pool() { static thread_local SplitPool* offer = nullptr; return offer; }

}  // namespace sb
