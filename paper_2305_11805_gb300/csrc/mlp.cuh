// Internal interface of the per-species network kernels.
#pragma once

#include "common.cuh"

namespace panna {

constexpr int kBM = 64, kBN = 64, kBK = 16;      // weight-gradient tiles (k_wgrad)
constexpr int kGM = 128, kGN = 128, kGK = 8;     // layer GEMM tiles (k_gemm): 256 threads, 8 x 8 outputs each
enum { PRO_NONE = 0, PRO_DACT = 1 };
enum { EPI_STORE = 0, EPI_FWD = 1, EPI_TAN = 2 };

// activations and their derivatives
__device__ __forceinline__ float act_f(int t, float z)
{
    switch (t) {
    case PANNA_ACT_GAUSSIAN: return __expf(-z * z);
    case PANNA_ACT_RELU: return z > 0.f ? z : 0.f;
    case PANNA_ACT_TANH: return tanhf(z);
    default: return z;
    }
}
__device__ __forceinline__ float act_d1(int t, float z)
{
    switch (t) {
    case PANNA_ACT_GAUSSIAN: return -2.f * z * __expf(-z * z);
    case PANNA_ACT_RELU: return z > 0.f ? 1.f : 0.f;
    case PANNA_ACT_TANH: { float h = tanhf(z); return 1.f - h * h; }
    default: return 1.f;
    }
}

// Per-species shape of one layer as a kernel argument.
struct LayerArgs {
    int S;
    int K[kMaxSpecies], N[kMaxSpecies], act[kMaxSpecies], pact[kMaxSpecies];
    int64_t w_off[kMaxSpecies], b_off[kMaxSpecies];
};

// Host-side description of all species' networks (same depth for every species).
struct MlpPlan {
    int S, L;
    int widths[kMaxSpecies][kMaxLayers + 1];
    int acts[kMaxSpecies][kMaxLayers];
    int64_t w_off[kMaxSpecies][kMaxLayers], b_off[kMaxSpecies][kMaxLayers];
    int ld[kMaxLayers + 1];   // row stride of layer-l activations = max width over species
    int64_t P;                // total parameters
    int max_hidden;           // max over l >= 1 of ld[l]
    int n_out;                // output width: 1 (energy) or 3 (charge equilibration)
    bool x3;                  // FP32 layer products on the tensor cores (mlp_x3.cu)
};

// Device buffers of one evaluation (rows in species order).
struct MlpBuffers {
    const float* G;                 // [N, ld[0]]
    float* Z[kMaxLayers + 1];       // pre-activations, l = 1..L
    float* A[kMaxLayers + 1];       // activations, l = 1..L
    float* Zd[kMaxLayers + 1];      // tangents
    float* Ad[kMaxLayers + 1];
    float* Ab; float* Ab2; float* Adb; float* Zb; float* Zdb;   // [N, max_hidden]
    float* part;                    // [splits, P]
    int splits;
    const int32_t* seg_off;
    int32_t* tile_start;
    DevStatus* status;
};

// One layer's product on the tensor cores from split FP32 operands (mlp_x3.cu); arguments of k_gemm
template <bool B_TRANS, int PRO, int EPI>
cudaError_t launch_gemm_x3(dim3 grid, cudaStream_t s, const LayerArgs& la, const float* theta, const int32_t* seg_off,
                           const int32_t* tile_start, const float* A, int lda, const float* Zp, int ldp, float* C,
                           int ldc, float* C2, const float* Ze, int lde, DevStatus* status);

cudaError_t mlp_tiles(const MlpPlan& p, const int32_t* seg_off, int32_t* tile_start, cudaStream_t s, int* launches);
cudaError_t mlp_forward(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, cudaStream_t s, int* launches);
cudaError_t mlp_energy_rows(const MlpPlan& p, const MlpBuffers& b, int64_t N, float* E_rows, cudaStream_t s, int* launches);
// g = dE/dG; seeded: b.Ab already holds the output seeds (rows, stride ld[L]) instead of dE/da_L = 1
cudaError_t mlp_input_grad(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, float* g,
                           cudaStream_t s, int* launches, bool seeded = false);
// Small batches (at most kSmallBatch rows, one output): forward pass, energies and, with g, the input
// gradient in one launch (mlp_small.cu); keep: Z and A of every layer are written as mlp_forward does.
// cudaErrorNotSupported for other batches and for networks too wide for its shared memory.
constexpr int64_t kSmallBatch = 2048;
cudaError_t mlp_small_rows(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, float* E_rows,
                           float* g, bool keep, cudaStream_t s, int* launches);
// BF16 tensor-core networks (mlp_tc.cu): energies and input gradients; ws from tc_workspace_bytes
size_t tc_workspace_bytes(const MlpPlan& p, int64_t N, bool split);
// g16_ready: the descriptor kernel already wrote the BF16 operand rows (tc_g16), else the FP32
// rows b.G are converted first
cudaError_t mlp_bf16_energy_grad(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, void* ws,
                                 bool split, float* E_rows, float* g, DevStatus* status, cudaStream_t s,
                                 int* launches, bool g16_ready = false);
// the BF16 descriptor operand rows (hi, lo; lo null without split) inside the workspace ws, or
// null when the descriptor width is not a multiple of 8
void tc_g16(const MlpPlan& p, int64_t N, bool split, void* ws, __nv_bfloat16** hi, __nv_bfloat16** lo);
// Parts of the weight-gradient pass: both (default); the forward tangent along wdot only (the
// output tangents land in b.Ad[L]); or the reverse pass only, with the output seeds already in
// b.Ab (energy part) and b.Adb (force part), rows of stride ld[L]
enum MlpGradPart { MLP_GRAD_ALL = 0, MLP_GRAD_TANGENT = 1, MLP_GRAD_REVERSE_SEEDED = 2 };
// wgrad_part (non-null: wgrad_workspace_bytes): the weight gradients on the tensor cores (wgrad_layer)
cudaError_t mlp_param_grad(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, const float* wdot,
                           const float* alpha_rows, float* dtheta, cudaStream_t s, int* launches,
                           float* wgrad_part = nullptr, MlpGradPart part = MLP_GRAD_ALL);

// Weight gradient of layer l + 1 (mlp_x3.cu): dW = Zb^T A + Zdb^T Ad, db = sum of Zb over the species'
// atoms, into dtheta.  A, Ad: the layer's inputs [N, ld[l]]; b.Zb, b.Zdb: its adjoints [N, ld[l + 1]]
size_t wgrad_workspace_bytes(const MlpPlan& p, int64_t N);
cudaError_t wgrad_layer(const MlpPlan& p, const MlpBuffers& b, int64_t N, float* part, int l, const LayerArgs& la,
                        const float* A, const float* Ad, float* dtheta, cudaStream_t s, int* launches);

// FP32 networks' products on the tensor cores (knob "mlp_fp32"): the layers' (forward, input gradient and
// tangents; either bit), the weight gradient's
enum { X3_LAYERS = 1 | 4, X3_WGRAD = 8 };

}  // namespace panna
