// Per-species networks (Eq. 1) on the 5th-generation tensor cores: BF16 operands, FP32 accumulation in
// tensor memory (TMEM), operands staged by TMA.  Operands may be carried as a hi + lo pair (three MMAs
// per product, hi*hi + hi*lo + lo*hi), which keeps about 16 significant bits.
//
// One GEMM kernel, C[rows, N] = A[rows, K] B_s[N, K]^T, serves every layer:
//   forward  Z_{l+1} = A_l W_l^T (+ b_l), A_{l+1} = act(Z_{l+1})       (B = W_l, K-major)
//   backward abar_l  = zbar_{l+1} W_l,   zbar_l = abar_l * act'(Z_l)    (B = W_l^T, K-major)
//            g       = zbar_1 W_0  (input gradient dE/dG, FP32 out)
// Rows are atoms in species order; a CTA owns one 128-row tile of one species (tile
// table on the device) and one N tile of up to 256 columns.
//
// CTA of 10 warps: warp 0 issues TMA loads into a 2-4 stage ring (mbarrier full/empty),
// warp 1 owns the TMEM allocation and one lane issues tcgen05.mma (M = 128, N = BN,
// K = 16 per instruction, 4 per 128-byte K chunk) and tcgen05.commit; warps 2..9
// read the accumulator with tcgen05.ld (two warps per 32-lane quarter) and run the epilogue.
// Every wait is bounded: on time-out the CTA sets PANNA_ERR_TIMEOUT, drains what it
// issued, frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>
#include <stdint.h>
#include <algorithm>
#include <string.h>

#include "mlp.cuh"
#include "tc.cuh"

namespace panna {

namespace {

constexpr int kTcBM = 128, kTcBK = 64;   // kTcBK: elements per 128-byte K chunk
constexpr int kTcEpiWarps = 8;                          // two per TMEM lane quarter
constexpr int kTcThreads = 64 + 32 * kTcEpiWarps;
constexpr uint32_t kTmemCols = 256;
constexpr uint32_t kTileA = kTcBM * kTcBK * 2;           // 16 KiB: one 128 x 64 BF16 tile

// Pipeline geometry by the number of parts each operand is carried in:
//   1: plain, N tile up to 256, 4 stages;
//   2: hi + lo (three MMAs per K step), N tile up to 128, 3 stages.
template <int PARTS>
struct TcCfg {
    static constexpr int kMaxBN = PARTS == 1 ? 256 : 128;
    static constexpr int kStages = PARTS == 1 ? 4 : 3;
    static constexpr int kParts = PARTS;
    static constexpr uint32_t kStageA = kParts * kTileA;
    static constexpr uint32_t kTileB = kMaxBN * kTcBK * 2;
    static constexpr uint32_t kStageB = kParts * kTileB;
    // with a 2 KB staging tile per epilogue warp for the FP32 outputs
    static constexpr size_t kSmem = 1024 + kStages * (kStageA + kStageB) + 256 + 2048 * 8;
};

enum { TC_FWD = 1, TC_BWD_MID = 2, TC_BWD_OUT = 3 };

// TMA descriptors of the parts of both operands (one kernel parameter in param space)
struct TcMaps {
    CUtensorMap a[2];
    CUtensorMap b[2];
};

struct TcArgs {
    int S;
    int N[kMaxSpecies];        // valid output columns per species
    int K;                     // reduction length (TMA zero-fills past the tensor edge)
    int BN;                    // N tile, multiple of 16, <= 256
    int n_pad;                 // rows per species in the stacked B operand
    int act[kMaxSpecies];      // FWD: activation of this layer; BWD_MID: of the layer whose Z is read
    const float* bias;         // FWD: [S * n_pad]
    float* outF; int ldF;      // FWD: Z (FP32); BWD_OUT: g (FP32)
    __nv_bfloat16* outH; int ldH;  // FWD: act(Z); BWD_MID: zbar (BF16, hi part when split)
    __nv_bfloat16* outL;           // split: lo part, same layout as outH
    const float* Zin; int ldZ;     // BWD_MID: Z for act'
    const int32_t* seg_off;
    const int32_t* tile_start;
    DevStatus* status;
};

__device__ __forceinline__ void store_split(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t idx, float v)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    hi[idx] = h;
    if (lo) lo[idx] = __float2bfloat16_rn(v - __bfloat162float(h));
}

// ------------------------------------------------------------------ helper kernels

__global__ void k_tiles128(int S, const int32_t* __restrict__ seg_off, int32_t* __restrict__ tile_start)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        int t = 0;
        for (int s = 0; s < S; ++s) {
            tile_start[s] = t;
            t += (seg_off[s + 1] - seg_off[s] + kTcBM - 1) / kTcBM;
        }
        tile_start[S] = t;
    }
}

__global__ void k_to_bf16(int64_t n, const float* __restrict__ x, __nv_bfloat16* __restrict__ hi,
                          __nv_bfloat16* __restrict__ lo)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) store_split(hi, lo, i, x[i]);
}

// Stacked weights of layer l for all species (BF16 hi + lo):
//   fwd: out[(s*npad + n) * kpad + k] = W_s[n][k]      (n < n_out_s, k < n_in_s, else 0)
//   bwd: out[(s*npad + k) * kpad + n] = W_s[n][k]      (the transpose)
__global__ void k_stack_weights(LayerArgs la, const float* __restrict__ theta, int npad, int kpad, int transpose,
                                __nv_bfloat16* __restrict__ out, __nv_bfloat16* __restrict__ out_lo,
                                float* __restrict__ bias_out)
{
    const int64_t total = (int64_t)la.S * npad * kpad;
    int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= total) return;
    const int s = (int)(idx / ((int64_t)npad * kpad));
    const int rr = (int)((idx / kpad) % npad);
    const int cc = (int)(idx % kpad);
    const int n_out = la.N[s], n_in = la.K[s];
    const int n = transpose ? cc : rr, k = transpose ? rr : cc;
    float v = 0.f;
    if (n < n_out && k < n_in) v = theta[la.w_off[s] + (int64_t)n * n_in + k];
    store_split(out, out_lo, idx, v);
    if (bias_out && !transpose && cc == 0) bias_out[(int64_t)s * npad + rr] = rr < n_out ? theta[la.b_off[s] + rr] : 0.f;
}

// Output layer (width 1) and the start of the backward pass, one warp per row:
//   z = sum_h w[h] act(Z[h]) + b, E = act_out(z), zbar[h] = act_out'(z) w[h] act'(Z[h]).
__global__ void k_out_layer(int S, const int32_t* __restrict__ seg_off, int64_t N, LayerArgs lo,
                            const float* __restrict__ theta,
                            const float* __restrict__ Z, int ldZ, float* __restrict__ E_rows,
                            __nv_bfloat16* __restrict__ zbar, __nv_bfloat16* __restrict__ zbar_lo, int ldzb,
                            LayerArgs lp)
{
    const int lane = threadIdx.x & 31;
    const int64_t r = (int64_t)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
    if (r >= N || r >= seg_off[S]) return;     // rows past the last species (ghost atoms have none)
    int s = 0;
    while (s < S - 1 && r >= seg_off[s + 1]) ++s;
    const int H = lo.K[s];
    const float* w = theta + lo.w_off[s];
    const int ta = lp.act[s];
    float acc = 0.f;
    for (int h = lane; h < H; h += 32) acc = fmaf(w[h], act_f(ta, Z[r * ldZ + h]), acc);
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    const float z = acc + theta[lo.b_off[s]];
    const int to = lo.act[s];
    if (lane == 0) E_rows[r] = act_f(to, z);
    const float dz = act_d1(to, z);
    for (int h = lane; h < ldzb; h += 32) {
        float v = 0.f;
        if (h < H) v = dz * w[h] * act_d1(ta, Z[r * ldZ + h]);
        store_split(zbar, zbar_lo, r * ldzb + h, v);
    }
}

// ------------------------------------------------------------------ host side

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encoder()
{
    if (g_encode) return cudaSuccess;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
    return cudaSuccess;
}

// 2D tensor [rows x cols] (row stride ld elements) of BF16 (box [box_rows x 64]): 128-byte rows, 128 B
// swizzle
cudaError_t make_map(CUtensorMap* m, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows)
{
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld * 2) % 16) return cudaErrorInvalidValue;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)(rows > 0 ? rows : 1)};
    cuuint64_t strides[1] = {(cuuint64_t)(ld * 2)};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                          const_cast<void*>(base), dims, strides, box, estr,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                          CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

int round_up(int x, int m) { return (x + m - 1) / m * m; }

LayerArgs tc_layer_args(const MlpPlan& p, int l)
{
    LayerArgs la{};
    la.S = p.S;
    for (int s = 0; s < p.S; ++s) {
        la.K[s] = p.widths[s][l];
        la.N[s] = p.widths[s][l + 1];
        la.act[s] = p.acts[s][l];
        la.pact[s] = p.acts[s][l];
        la.w_off[s] = p.w_off[s][l];
        la.b_off[s] = p.b_off[s][l];
    }
    return la;
}

int tc_bn(int n, int max_bn) { int t = (n + max_bn - 1) / max_bn; return round_up((n + t - 1) / t, 16); }

// Persistent form of the row-tiled GEMM for the BF16 networks' layers (TC_FWD, TC_BWD_MID,
// TC_BWD_OUT).  One CTA per SM walks the work items (128-row tile of one species x N tile)
// with a stride of the grid size.  The TMA warp runs ahead through the stage ring across item
// boundaries; the MMA warp alternates between two TMEM accumulators, so the epilogue warps
// drain item j (tcgen05.ld, bias / activation, stores straight from registers: each thread
// writes whole 32-byte sectors of its own row) while the MMAs of item j + 1 run.  Barriers:
// full / empty per stage (TMA <-> MMA), acc_full / acc_empty per accumulator (MMA <->
// epilogue, the latter counting one arrival per epilogue warp).  Every wait is bounded.
__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

struct ItemPos {
    int s, row0, rend, n0;
    bool valid;
};

__device__ __forceinline__ ItemPos tc_item(const TcArgs& a, int item, int n_nt)
{
    ItemPos p;
    const int tile = item / n_nt, nt = item - tile * n_nt;
    int s = 0;
    while (tile >= a.tile_start[s + 1]) ++s;
    p.s = s;
    p.n0 = nt * a.BN;
    p.row0 = a.seg_off[s] + (tile - a.tile_start[s]) * kTcBM;
    p.rend = a.seg_off[s + 1];
    p.valid = p.n0 < a.N[s];
    return p;
}

template <int EPI, int PARTS>
__global__ void __launch_bounds__(kTcThreads, 1)
k_tc_gemm_p(const __grid_constant__ TcMaps tm, TcArgs a, int n_nt)
{
    using Cfg = TcCfg<PARTS>;
    constexpr int kStages = Cfg::kStages;
    constexpr int BKE = kTcBK;                           // BF16 elements per 128-byte K chunk
    constexpr int MMAK = 16;                             // K per instruction
    constexpr uint32_t kAcc = Cfg::kMaxBN;               // TMEM columns per accumulator
    extern __shared__ unsigned char smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sA = smem;
    uint8_t* sB = smem + kStages * Cfg::kStageA;
    uint64_t* full = reinterpret_cast<uint64_t*>(sB + kStages * Cfg::kStageB);
    uint64_t* empty = full + kStages;
    uint64_t* accf = empty + kStages;                    // [2]
    uint64_t* acce = accf + 2;                           // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    // FP32 output staging, 2 KB per epilogue warp, past the barriers (kSmemP - kSmem bytes)
    float* stg = reinterpret_cast<float*>(sB + kStages * Cfg::kStageB + 256);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_items = a.tile_start[a.S] * n_nt;
    const int nk = (a.K + BKE - 1) / BKE;
    if (threadIdx.x == 0) {
        for (int i = 0; i < kStages; ++i) { mbar_init(full + i, 1); mbar_init(empty + i, 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(accf + i, 1); mbar_init(acce + i, kTcEpiWarps); }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) tmem_alloc(tmem_slot, 2 * kAcc);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const uint32_t bytes = Cfg::kParts * (kTileA + (uint32_t)a.BN * 128u);

    if (warp == 0) {
        if (lane == 0) {
            int g = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const ItemPos ip = tc_item(a, item, n_nt);
                if (!ip.valid) continue;
                for (int kc = 0; kc < nk; ++kc, ++g) {
                    const int st = g % kStages;
                    const uint32_t ph = (uint32_t)(g / kStages) & 1u;
                    if (!mbar_wait(empty + st, ph ^ 1u, abort_flag)) { *abort_flag = 1; ok = false; break; }
                    mbar_expect_tx(full + st, bytes);
                    uint8_t* a_st = sA + st * Cfg::kStageA;
                    uint8_t* b_st = sB + st * Cfg::kStageB;
#pragma unroll
                    for (int q = 0; q < PARTS; ++q) {
                        tma_load_2d(a_st + q * kTileA, &tm.a[q], kc * BKE, ip.row0, full + st);
                        tma_load_2d(b_st + q * Cfg::kTileB, &tm.b[q], kc * BKE, ip.s * a.n_pad + ip.n0, full + st);
                    }
                }
            }
            // never leave with copies in flight
            for (int k = g > kStages ? g - kStages : 0; k < g; ++k)
                mbar_wait(full + k % kStages, (uint32_t)(k / kStages) & 1u, nullptr);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            const uint32_t idesc = idesc_mma(false, kTcBM, (uint32_t)a.BN);
            int g = 0, j = 0;
            bool ok = true;
            for (int item = blockIdx.x; item < n_items && ok; item += gridDim.x) {
                const ItemPos ip = tc_item(a, item, n_nt);
                if (!ip.valid) continue;
                const int b = j & 1;
                if (!mbar_wait(acce + b, ((uint32_t)(j >> 1) & 1u) ^ 1u, abort_flag)) { *abort_flag = 1; break; }
                tc_fence_after();
                const uint32_t d = tmem + (uint32_t)b * kAcc;
                for (int kc = 0; kc < nk; ++kc, ++g) {
                    const int st = g % kStages;
                    const uint32_t ph = (uint32_t)(g / kStages) & 1u;
                    if (!mbar_wait(full + st, ph, abort_flag)) { *abort_flag = 1; ok = false; break; }
                    tc_fence_after();
                    const uint32_t a0 = smem_u32(sA + st * Cfg::kStageA), b0 = smem_u32(sB + st * Cfg::kStageB);
#pragma unroll
                    for (int kk = 0; kk < BKE / MMAK; ++kk) {
                        const uint64_t a1 = sw128_desc(a0 + kk * 32), b1 = sw128_desc(b0 + kk * 32);
                        tc_mma(d, a1, b1, idesc, (kc | kk) ? 1u : 0u);
                        if (PARTS >= 2) {
                            const uint64_t a2 = sw128_desc(a0 + kTileA + kk * 32);
                            const uint64_t b2 = sw128_desc(b0 + Cfg::kTileB + kk * 32);
                            tc_mma(d, a1, b2, idesc, 1u);
                            tc_mma(d, a2, b1, idesc, 1u);
                        }
                    }
                    tc_commit(empty + st);
                }
                tc_commit(accf + b);   // arrives once the item's MMAs have completed
                ++j;
            }
            // no TMEM release under running MMAs: the epilogue waited for every committed item;
            // after an abort wait (bounded) for whatever was issued last
            if (!ok || *abort_flag) {
                tc_commit(accf + (j & 1));
                mbar_wait(accf + (j & 1), ((uint32_t)(j >> 1) & 1u), nullptr);
            }
        }
    } else {
        const int ew = warp - 2;
        const int q = warp & 3;                    // TMEM lane quarter of this warp
        const int half = ew >> 2;
        int j = 0;
        for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
            const ItemPos ip = tc_item(a, item, n_nt);
            if (!ip.valid) continue;
            const int b = j & 1;
            const int r = ip.row0 + q * 32 + lane;
            const bool row_ok = r < ip.rend;
            const int s = ip.s, Ns = a.N[s];
            // BWD_MID: the pre-activations of the next 16 columns are loaded one chunk ahead (the
            // first before the wait for the MMAs), so their latency overlaps the TMEM wait and the
            // previous chunk's arithmetic and stores
            float zn[16];
            auto load_z = [&](int c) {
                const int n = ip.n0 + c;
                if (EPI != TC_BWD_MID || !row_ok || c >= a.BN || n >= Ns) return;
                const float* z = a.Zin + (size_t)r * a.ldZ + n;
                if (n + 16 <= Ns && (reinterpret_cast<uintptr_t>(z) & 15) == 0) {
#pragma unroll
                    for (int k = 0; k < 16; k += 4) {
                        const float4 t4 = *reinterpret_cast<const float4*>(z + k);
                        zn[k] = t4.x; zn[k + 1] = t4.y; zn[k + 2] = t4.z; zn[k + 3] = t4.w;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) zn[k] = (n + k < Ns) ? z[k] : 0.f;
                }
            };
            load_z(half * 16);
            if (!mbar_wait(accf + b, (uint32_t)(j >> 1) & 1u, abort_flag)) { *abort_flag = 1; break; }
            tc_fence_after();
            for (int c0 = half * 16; c0 < a.BN; c0 += 32) {
                float v[16];
                tc_ld16(tmem + (uint32_t)b * kAcc + ((uint32_t)(q * 32) << 16) + (uint32_t)c0, v);
                const int n = ip.n0 + c0;
                if (n >= Ns) continue;   // the same for the whole warp
                const bool whole = n + 16 <= Ns;
                float zv[16];
                if (EPI == TC_BWD_MID) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) zv[k] = zn[k];
                    load_z(c0 + 32);
                }
                float o1[16], o2[16];
                if (EPI == TC_FWD) {
                    const float* bias = a.bias + s * a.n_pad + n;
                    float bv[16];
                    if ((reinterpret_cast<uintptr_t>(bias) & 15) == 0) {
#pragma unroll
                        for (int k = 0; k < 16; k += 4) {
                            const float4 t4 = *reinterpret_cast<const float4*>(bias + k);
                            bv[k] = t4.x; bv[k + 1] = t4.y; bv[k + 2] = t4.z; bv[k + 3] = t4.w;
                        }
                    } else {
#pragma unroll
                        for (int k = 0; k < 16; ++k) bv[k] = bias[k];
                    }
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        o1[k] = v[k] + bv[k];
                        o2[k] = act_f(a.act[s], o1[k]);
                    }
                } else if (EPI == TC_BWD_MID) {
#pragma unroll
                    for (int k = 0; k < 16; ++k) o2[k] = (whole || n + k < Ns) ? v[k] * act_d1(a.act[s], zv[k]) : 0.f;
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k) o1[k] = v[k];
                }
                if (EPI == TC_FWD || EPI == TC_BWD_OUT) {
                    const bool aligned = (a.ldF & 3) == 0 &&
                                         (reinterpret_cast<uintptr_t>(a.outF + (size_t)ip.row0 * a.ldF + n) & 15) == 0;
                    if (whole && aligned) {
                        // through the warp's staging tile: each lane writes its row's 16 values
                        // (16-byte pieces swizzled by row, conflict-free), then the warp stores
                        // 8 rows x 64 contiguous bytes per instruction instead of 32 rows x 16
                        float* st = stg + ew * 512;
                        const int sw = (lane >> 1) & 3;
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            *reinterpret_cast<float4*>(st + lane * 16 + 4 * (k ^ sw)) =
                                make_float4(o1[4 * k], o1[4 * k + 1], o1[4 * k + 2], o1[4 * k + 3]);
                        __syncwarp();
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const int row = i * 8 + (lane >> 2), pc = lane & 3;
                            const float4 val = *reinterpret_cast<const float4*>(st + row * 16 + 4 * (pc ^ ((row >> 1) & 3)));
                            const int rr = ip.row0 + q * 32 + row;
                            if (rr < ip.rend)
                                *reinterpret_cast<float4*>(a.outF + (size_t)rr * a.ldF + n + 4 * pc) = val;
                        }
                        __syncwarp();
                    } else if (row_ok) {
                        float* o = a.outF + (size_t)r * a.ldF + n;
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            if (n + k < Ns) o[k] = o1[k];
                    }
                }
                if (EPI == TC_FWD || EPI == TC_BWD_MID) {
                    const bool aligned = (a.ldH & 7) == 0 &&
                                         (reinterpret_cast<uintptr_t>(a.outH + (size_t)ip.row0 * a.ldH + n) & 15) == 0 &&
                                         (PARTS < 2 ||
                                          (reinterpret_cast<uintptr_t>(a.outL + (size_t)ip.row0 * a.ldH + n) & 15) == 0);
                    if (whole && aligned) {
                        uint32_t hw[8], lw[8];
#pragma unroll
                        for (int k = 0; k < 16; k += 2) {
                            const __nv_bfloat16 h0 = __float2bfloat16_rn(o2[k]), h1 = __float2bfloat16_rn(o2[k + 1]);
                            const __nv_bfloat16 l0 = __float2bfloat16_rn(o2[k] - __bfloat162float(h0));
                            const __nv_bfloat16 l1 = __float2bfloat16_rn(o2[k + 1] - __bfloat162float(h1));
                            hw[k / 2] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
                            lw[k / 2] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
                        }
                        // through the staging tile: hi rows then lo rows, 32 B per row, the two
                        // 16-byte pieces swapped on every other group of four rows (conflict-free);
                        // the warp then stores 16 rows x 32 contiguous bytes per instruction
                        uint4* st = reinterpret_cast<uint4*>(stg + ew * 512);
                        const int sw = (lane >> 2) & 1;
                        st[lane * 2 + (0 ^ sw)] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
                        st[lane * 2 + (1 ^ sw)] = make_uint4(hw[4], hw[5], hw[6], hw[7]);
                        if (PARTS >= 2) {
                            st[64 + lane * 2 + (0 ^ sw)] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
                            st[64 + lane * 2 + (1 ^ sw)] = make_uint4(lw[4], lw[5], lw[6], lw[7]);
                        }
                        __syncwarp();
#pragma unroll
                        for (int part = 0; part < (PARTS >= 2 ? 2 : 1); ++part) {
                            __nv_bfloat16* base = part ? a.outL : a.outH;
#pragma unroll
                            for (int i = 0; i < 2; ++i) {
                                const int row = i * 16 + (lane >> 1), pc = lane & 1;
                                const uint4 val = st[part * 64 + row * 2 + (pc ^ ((row >> 2) & 1))];
                                const int rr = ip.row0 + q * 32 + row;
                                if (rr < ip.rend)
                                    *reinterpret_cast<uint4*>(base + (size_t)rr * a.ldH + n + 8 * pc) = val;
                            }
                        }
                        __syncwarp();
                    } else if (row_ok) {
#pragma unroll
                        for (int k = 0; k < 16; ++k)
                            if (n + k < Ns)
                                store_split(a.outH, PARTS >= 2 ? a.outL : nullptr, (size_t)r * a.ldH + n + k, o2[k]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acce + b);
            ++j;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && *abort_flag) set_status(a.status, PANNA_ERR_TIMEOUT, blockIdx.x);
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, 2 * kAcc);
    }
}

// persistent launch: one CTA per SM (at most one per work item)
template <int EPI, int PARTS>
cudaError_t launch_tc_p(const TcMaps& m, const TcArgs& ta, int64_t N, int nmax, cudaStream_t s)
{
    static int n_sm = 0;
    if (n_sm == 0) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
    }
    const int n_nt = (nmax + ta.BN - 1) / ta.BN;
    const int64_t items = ((N + kTcBM - 1) / kTcBM + ta.S) * n_nt;
    const unsigned grid = (unsigned)std::min<int64_t>(items, n_sm);
    const int smem = (int)TcCfg<PARTS>::kSmem;
    cudaError_t e = allow_smem(k_tc_gemm_p<EPI, PARTS>, smem);
    if (e != cudaSuccess) return e;
    k_tc_gemm_p<EPI, PARTS><<<grid, kTcThreads, smem, s>>>(m, ta, n_nt);
    return cudaGetLastError();
}

template <int EPI>
cudaError_t launch_tc_any(bool split, const TcMaps& m, const TcArgs& ta, int64_t N, int nmax, cudaStream_t s)
{
    return split ? launch_tc_p<EPI, 2>(m, ta, N, nmax, s) : launch_tc_p<EPI, 1>(m, ta, N, nmax, s);
}

// Buffers of the BF16 networks, carved from one workspace block (sizing when base == nullptr).
struct TcBufs {
    int32_t* tiles128;
    __nv_bfloat16* G16[2];                       // hi, lo
    __nv_bfloat16* A16[kMaxLayers + 1][2];
    __nv_bfloat16* Zb16[kMaxLayers + 1][2];
    __nv_bfloat16* Wf[kMaxLayers][2];
    __nv_bfloat16* Wb[kMaxLayers][2];
    float* bias[kMaxLayers];
    int ldh[kMaxLayers + 1];
    int npf[kMaxLayers], npb[kMaxLayers], bnf[kMaxLayers], bnb[kMaxLayers];
};

size_t tc_carve(const MlpPlan& p, int64_t N, bool split, char* base, TcBufs& t)
{
    size_t off = 0;
    auto take = [&](size_t n) {
        void* q = base ? base + off : nullptr;
        off += (n + 255) & ~(size_t)255;
        return q;
    };
    const int parts = split ? 2 : 1;
    const int max_bn = split ? TcCfg<2>::kMaxBN : TcCfg<1>::kMaxBN;
    t.tiles128 = static_cast<int32_t*>(take((kMaxSpecies + 1) * sizeof(int32_t)));
    t.ldh[0] = round_up(p.ld[0], 8);
    for (int q = 0; q < 2; ++q) t.G16[q] = q < parts ? static_cast<__nv_bfloat16*>(take((size_t)N * t.ldh[0] * 2)) : nullptr;
    for (int l = 1; l < p.L; ++l) {
        t.ldh[l] = round_up(p.ld[l], 8);
        for (int q = 0; q < 2; ++q) {
            t.A16[l][q] = q < parts ? static_cast<__nv_bfloat16*>(take((size_t)N * t.ldh[l] * 2)) : nullptr;
            t.Zb16[l][q] = q < parts ? static_cast<__nv_bfloat16*>(take((size_t)N * t.ldh[l] * 2)) : nullptr;
        }
    }
    for (int l = 0; l < p.L - 1; ++l) {
        const int no = p.ld[l + 1], ni = p.ld[l];
        t.bnf[l] = tc_bn(no, max_bn); t.bnb[l] = tc_bn(ni, max_bn);
        t.npf[l] = round_up(no, t.bnf[l]); t.npb[l] = round_up(ni, t.bnb[l]);
        for (int q = 0; q < 2; ++q) {
            t.Wf[l][q] = q < parts ? static_cast<__nv_bfloat16*>(take((size_t)p.S * t.npf[l] * round_up(ni, 8) * 2)) : nullptr;
            t.Wb[l][q] = q < parts ? static_cast<__nv_bfloat16*>(take((size_t)p.S * t.npb[l] * round_up(no, 8) * 2)) : nullptr;
        }
        t.bias[l] = static_cast<float*>(take((size_t)p.S * t.npf[l] * 4));
    }
    return off + 4096;
}

// 2D BF16 tensor [rows x cols] (row stride ld elements), box [box_rows x 64], 128 B swizzle
cudaError_t make_maps(CUtensorMap* m, __nv_bfloat16* const* base, int parts, int64_t rows, int64_t cols, int64_t ld,
                      int box_rows)
{
    for (int q = 0; q < parts; ++q) {
        cudaError_t e = make_map(&m[q], base[q], rows, cols, ld, box_rows);
        if (e != cudaSuccess) return e;
    }
    if (parts == 1) m[1] = m[0];
    return cudaSuccess;
}

}  // namespace

size_t tc_workspace_bytes(const MlpPlan& p, int64_t N, bool split)
{
    TcBufs t;
    return tc_carve(p, N, split, nullptr, t);
}

// Energies (E_rows) and input gradients g = dE/dG (FP32 rows) of all rows with BF16 tensor-core
// GEMMs (FP32 accumulation).  split: every BF16 operand is carried as a hi + lo pair and each
// product takes three MMAs (hi*hi + hi*lo + lo*hi), about 16 significant bits per operand.
// G rows in FP32 are converted first.  Needs at least one hidden layer.
void tc_g16(const MlpPlan& p, int64_t N, bool split, void* ws, __nv_bfloat16** hi, __nv_bfloat16** lo)
{
    TcBufs t;
    tc_carve(p, N, split, static_cast<char*>(ws), t);
    *hi = t.ldh[0] == p.ld[0] ? t.G16[0] : nullptr;
    *lo = t.ldh[0] == p.ld[0] ? t.G16[1] : nullptr;
}

cudaError_t mlp_bf16_energy_grad(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, void* ws,
                                 bool split, float* E_rows, float* g, DevStatus* status, cudaStream_t s,
                                 int* launches, bool g16_ready)
{
    if (p.L < 2) return cudaErrorNotSupported;
    cudaError_t e = get_encoder();
    if (e != cudaSuccess) return e;
    TcBufs t;
    tc_carve(p, N, split, static_cast<char*>(ws), t);
    const int parts = split ? 2 : 1;
    if (t.ldh[0] != p.ld[0]) return cudaErrorNotSupported;   // descriptor width not a multiple of 8
    k_tiles128<<<1, 32, 0, s>>>(p.S, b.seg_off, t.tiles128);
    ++*launches;
    for (int l = 0; l < p.L - 1; ++l) {
        const int no = p.ld[l + 1], ni = p.ld[l];
        LayerArgs la = tc_layer_args(p, l);
        int64_t tf = (int64_t)p.S * t.npf[l] * round_up(ni, 8);
        k_stack_weights<<<(unsigned)((tf + 255) / 256), 256, 0, s>>>(la, theta, t.npf[l], round_up(ni, 8), 0,
                                                                    t.Wf[l][0], t.Wf[l][1], t.bias[l]);
        int64_t tb = (int64_t)p.S * t.npb[l] * round_up(no, 8);
        k_stack_weights<<<(unsigned)((tb + 255) / 256), 256, 0, s>>>(la, theta, t.npb[l], round_up(no, 8), 1,
                                                                    t.Wb[l][0], t.Wb[l][1], nullptr);
        *launches += 2;
    }
    // padding columns of the BF16 operands meet zero weights, but must not hold NaN (the
    // epilogues write the species' own columns only); layers without padding need no clearing
    for (int l = 1; l < p.L; ++l) {
        bool pad = false;
        for (int q = 0; q < p.S; ++q) pad = pad || p.widths[q][l] != t.ldh[l];
        if (!pad) continue;
        for (int q = 0; q < parts; ++q) {
            e = cudaMemsetAsync(t.A16[l][q], 0, (size_t)N * t.ldh[l] * 2, s);
            if (e == cudaSuccess) e = cudaMemsetAsync(t.Zb16[l][q], 0, (size_t)N * t.ldh[l] * 2, s);
            if (e != cudaSuccess) return e;
        }
    }
    if (!g16_ready) {
        k_to_bf16<<<(unsigned)((N * t.ldh[0] + 255) / 256), 256, 0, s>>>(N * t.ldh[0], b.G, t.G16[0], t.G16[1]);
        ++*launches;
    }

    TcArgs base{};
    base.S = p.S;
    base.seg_off = b.seg_off;
    base.tile_start = t.tiles128;
    base.status = status;
    TcMaps maps;
    // forward through the hidden layers
    for (int l = 0; l < p.L - 1; ++l) {
        CUtensorMap mA[2], mB[2];
        __nv_bfloat16* const* Ain = l == 0 ? t.G16 : t.A16[l];
        e = make_maps(mA, Ain, parts, N, p.ld[l], t.ldh[l], kTcBM);
        if (e == cudaSuccess)
            e = make_maps(mB, t.Wf[l], parts, (int64_t)p.S * t.npf[l], p.ld[l], round_up(p.ld[l], 8), t.bnf[l]);
        if (e != cudaSuccess) return e;
        maps.a[0] = mA[0]; maps.b[0] = mB[0]; maps.a[1] = mA[1]; maps.b[1] = mB[1];
        TcArgs ta = base;
        for (int q = 0; q < p.S; ++q) { ta.N[q] = p.widths[q][l + 1]; ta.act[q] = p.acts[q][l]; }
        ta.K = p.ld[l];
        ta.BN = t.bnf[l];
        ta.n_pad = t.npf[l];
        ta.bias = t.bias[l];
        ta.outF = b.Z[l + 1]; ta.ldF = p.ld[l + 1];
        ta.outH = t.A16[l + 1][0]; ta.outL = t.A16[l + 1][1]; ta.ldH = t.ldh[l + 1];
        e = launch_tc_any<TC_FWD>(split, maps, ta, N, p.ld[l + 1], s);
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    // output layer and the first backward step
    {
        LayerArgs lo = tc_layer_args(p, p.L - 1);
        LayerArgs lp = tc_layer_args(p, p.L - 2);
        k_out_layer<<<(unsigned)((N + 7) / 8), 256, 0, s>>>(p.S, b.seg_off, N, lo, theta, b.Z[p.L - 1],
                                                           p.ld[p.L - 1], E_rows, t.Zb16[p.L - 1][0],
                                                           t.Zb16[p.L - 1][1], t.ldh[p.L - 1], lp);
        ++*launches;
    }
    // backward through the hidden layers down to the input gradient
    for (int l = p.L - 2; l >= 0; --l) {
        CUtensorMap mA[2], mB[2];
        e = make_maps(mA, t.Zb16[l + 1], parts, N, p.ld[l + 1], t.ldh[l + 1], kTcBM);
        if (e == cudaSuccess)
            e = make_maps(mB, t.Wb[l], parts, (int64_t)p.S * t.npb[l], p.ld[l + 1], round_up(p.ld[l + 1], 8),
                          t.bnb[l]);
        if (e != cudaSuccess) return e;
        maps.a[0] = mA[0]; maps.b[0] = mB[0]; maps.a[1] = mA[1]; maps.b[1] = mB[1];
        TcArgs ta = base;
        for (int q = 0; q < p.S; ++q) ta.N[q] = p.widths[q][l];
        ta.K = p.ld[l + 1];
        ta.BN = t.bnb[l];
        ta.n_pad = t.npb[l];
        if (l > 0) {
            for (int q = 0; q < p.S; ++q) ta.act[q] = p.acts[q][l - 1];
            ta.Zin = b.Z[l]; ta.ldZ = p.ld[l];
            ta.outH = t.Zb16[l][0]; ta.outL = t.Zb16[l][1]; ta.ldH = t.ldh[l];
            e = launch_tc_any<TC_BWD_MID>(split, maps, ta, N, p.ld[l], s);
        } else {
            ta.outF = g; ta.ldF = p.ld[0];
            e = launch_tc_any<TC_BWD_OUT>(split, maps, ta, N, p.ld[0], s);
        }
        if (e != cudaSuccess) return e;
        ++*launches;
    }
    return cudaGetLastError();
}

}  // namespace panna
