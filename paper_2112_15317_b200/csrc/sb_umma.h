// Interface between the host planner (sb_api.cu) and the tcgen05 tensor-core path (sb_umma.cu).
#pragma once

#include "../../include/splitbrain.h"
#include "sb_internal.h"
#include <cuda.h>

namespace sb {

// One planned tensor-core launch: tensor maps, tile geometry and epilogue pointers.
struct UmmaOp {
    bool enabled = false;
    alignas(64) CUtensorMap mapA;
    alignas(64) CUtensorMap mapB;
    alignas(64) CUtensorMap mapC;          // output tensor, for the TMA-store epilogue (when the op's tma_out is set);
                                           // FC weight gradient: the float master weights [out][in] (update folded in)
    alignas(64) CUtensorMap mapD;          // FC weight gradient: the momentum buffer, same shape
    alignas(16) unsigned char blob[512];   // kernel parameters, tile width and grid (see sb_umma.cu)
};
struct UmmaLayer {
    UmmaOp fwd, dgrad, wgrad;
    bool conv_in = false;                // input-layer conv on the tensor cores (wgrad.mapA then maps this layer's dy,
                                         // fwd.mapA its output for the TMA store)
    const void* bound_input = nullptr;   // layer 0 only: the input buffer the tensor maps currently point at
    bool pool_fused = false;             // conv layer followed by a 2x2 max-pool: the forward kernel also writes the pool layer's
                                         // output and argmax bytes from its staged output tile
};

// Read-only views of the model for the planner in sb_umma.cu.
struct ModelView {
    const sb_config* cfg;
    bool bf16;
    int B, n_layers, first_fc;
    float *Wm, *Gm, *Vm;
    __nv_bfloat16* Sm;
    float* ws;      // data-side scratch
    float* ws_wk[8];  // weight-side scratch regions, one per weight stream: layer i uses ws_wk[i % n_wstreams]
    int n_wstreams;   // 0: everything runs on the caller's stream (region 0)
    size_t ws_floats;
    uint32_t* status;
    char* input_grad;
    const PtrTab* x_tab;
    char* stage_x;        // contiguous [B, input] staging area inside the arena
};
struct LayerView {
    int kind, H, W, Cin, Cout, in_f, out_f;
    int K;                // FC: this layer's column shards
    bool relu;
    size_t p_w, p_b, n_w, n_b;
    char *act, *dact;
    unsigned char* pool_idx;   // pool layers: argmax bytes
    const char* in_act;   // previous layer's output (nullptr for layer 0)
    char* d_below;        // where the input gradient goes
    bool below_relu;
    UmmaLayer* um;
};
ModelView model_view(sb_model* m);
LayerView layer_view(sb_model* m, int i);
int64_t* launch_counter(sb_model* m);

// Scratch floats the tensor-core path needs (split partial sums); called during planning,
// before the arena exists (pointers in the views are null or unset).
sb_status umma_plan_scratch(sb_model* m, size_t* floats);
// Whether layer i's passes run on tensor-core tiles (the input layer's im2col kernels aside).
bool umma_layer_ok(sb_model* m, int layer);
// Encodes tensor maps and decides, per layer and pass, whether the tensor-core kernel runs (layers first_layer..).
sb_status umma_plan_layers(sb_model* m, int first_layer);

sb_status umma_conv_fwd(sb_model* m, int layer, cudaStream_t st);
sb_status umma_conv_dgrad(sb_model* m, int layer, cudaStream_t st);
// Launches the weight-gradient kernel; *splits > 1 means it wrote split partial sums at *part
// (to be reduced in split order by the caller), else it wrote the gradient itself.
sb_status umma_conv_wgrad_launch(sb_model* m, int layer, cudaStream_t st, int* splits, float** part);
// false: the layer's weight-gradient kernel (CTA-pair variant) leaves the bias gradient to a column-sum kernel
bool umma_wgrad_bias_fused(sb_model* m, int layer);
// First-layer FC: points the tensor maps that read the network input at `x` ([B, in] contiguous, bf16).
sb_status umma_bind_input(sb_model* m, const void* x);
sb_status umma_fc_fwd(sb_model* m, int layer, cudaStream_t st);
sb_status umma_fc_dgrad(sb_model* m, int layer, cudaStream_t st);
sb_status umma_fc_wgrad(sb_model* m, int layer, cudaStream_t st);
// FC weight gradient with the SGD-momentum update applied in the kernel's epilogue (gradient never stored): possible when
// umma_fc_wgrad_can_update says so (unsplit reduction, staged epilogue, bias gradient in the same kernel)
bool umma_fc_wgrad_can_update(sb_model* m, int layer);
sb_status umma_fc_wgrad_update(sb_model* m, int layer, Hyper hy, cudaStream_t st);

// Input-layer convolution (1, 3 or 4 input channels, 16, 32, 48 or 64 output channels, bf16) on the tensor cores.
bool conv_in_umma_supported(int H, int W, int Cin, int Cout);
// Partial buffers the weight-gradient kernel writes ([blocks][Cout*9*Cin + Cout] floats, reduced in block order).
int conv_in_umma_wgrad_blocks(int B, int H, int W, int Cin);
// mapY, mapDy: tensor maps of the output and of its gradient as [pixels][Cout] with (64, 128) boxes
cudaError_t launch_conv_in_fwd_umma(const ConvSimtArgs& a, const CUtensorMap& mapY, uint32_t* status, cudaStream_t st);
cudaError_t launch_conv_in_wgrad_umma(const WgradSimtArgs& a, const CUtensorMap& mapDy, uint32_t* status, cudaStream_t st);

// Weight gradient of a 3x3 layer with at most 64 channels on either side (sb_conv64_wgrad.cu).  The maps list the dimensions as
// (c, w, n, h) with boxes of (64, bw, bn, bh + 1); the box of a chunk holds 64 pixels, bw * bn a multiple of 8.
struct Conv64WgradArgs {
    const CUtensorMap *mapDy, *mapX;
    int bw, bh, bn, tiles_w, tiles_h, total_chunks, chunks_per_cta;
    int Cin, Cout;
    float* out;                      // one partial gradient per CTA, split_stride floats apart; 16-byte aligned, as is split_stride
    long split_stride, bias_off;
    uint32_t* status;
};
int conv64_wgrad_stages(int bw, int bh, int bn);      // ring depth that fits (at least 2 for the kernel to run)
cudaError_t launch_conv64_wgrad(const Conv64WgradArgs& a, cudaStream_t st);

// Stored weight gradient of a large FC layer (sb_fc_wgrad.cu); maps with boxes of 64 columns x 64 batch rows.
struct FcWgradArgs {
    const CUtensorMap *mapDy, *mapX;
    int batch, out_f, in_f;
    float *out, *bias;               // 16-byte aligned, in_f a multiple of 4
    uint32_t* status;
};
cudaError_t launch_fc_wgrad(const FcWgradArgs& a, cudaStream_t st);

// Tensor map of a row-major float matrix with boxes of 32 columns x box_rows rows: rows of 128 bytes in the 128-byte swizzle.
bool umma_map_f32_rows(CUtensorMap* map, const void* ptr, long rows, long cols, int box_rows);
// Tensor map of three row-major bf16 matrices, plane_stride elements apart, with boxes of 64 columns x box_rows rows of one plane.
bool umma_map_terms(CUtensorMap* map, const void* ptr, long rows, long cols, size_t plane_stride, int box_rows);

const char* umma_last_error();
// One CTA that waits (bounded by limit_ns) on a barrier nothing completes, then reports through the status word.
cudaError_t launch_wait_probe(uint32_t* status, unsigned long long limit_ns, cudaStream_t st);
#ifdef SB_CTA_TIMING
// Development builds only: when set to a device buffer of 1024*16 uint64, every tensor-core CTA (first 1024 of a launch)
// records clock stamps at its phase boundaries.
void umma_set_timing_buffer(void* dev_ptr);
void umma_set_trace_buffer(void* dev_ptr);
#endif

}  // namespace sb
