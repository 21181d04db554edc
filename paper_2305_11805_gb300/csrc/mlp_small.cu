// Per-species networks of a small batch in one launch: forward pass, atomic energies and input gradients
// dE/dG of all layers, FP32 on the CUDA cores.
//
// For a few hundred atoms the layer-by-layer GEMMs of mlp.cu fill one to a dozen CTAs, each of which
// walks its reduction alone: latency, not arithmetic, decides (a 64-atom box with a 96-256-128-32-1
// network: ten launches, 140 us).  Here a CTA takes R rows of one species through every layer with the
// activations in shared memory and the weights read from L2.  Forward, a warp owns four output units
// and its lanes share the reduction, 16 bytes of each weight row per lane (whole lines); the 4 x R sums
// meet in one butterfly.  Backward, a warp owns 128 inputs and a slice of the units; the slices' sums
// meet in shared memory in a fixed order.
//
// The weights cross from L2 once per CTA, so the time grows with N / R.  Measured (forward + energies + input
// gradient, us, here / layer by layer with k_gemm_x3 just past the line of 2,048 rows): 64 rows of
// 96-256-128-32-1 28; 768-128-32-1: 850 rows 47, 1,960 rows 82 / 2,200 rows 103; 256-256-128-1: 2,000 rows 78 /
// 2,052 rows 107; 192-128-64-1: 2,048 rows 45 / 2,916 rows 78.
#include <algorithm>

#include "mlp.cuh"

namespace panna {

namespace {

constexpr int kRowThreads = 512, kRowWarps = kRowThreads / 32;

struct NetDev {
    int S, L;
    int widths[kMaxSpecies][kMaxLayers + 1];
    int acts[kMaxSpecies][kMaxLayers];
    int64_t w_off[kMaxSpecies][kMaxLayers], b_off[kMaxSpecies][kMaxLayers];
    int ld[kMaxLayers + 1];
    float* Z[kMaxLayers + 1];
    float* A[kMaxLayers + 1];
};

// four consecutive values of a row of length n from index k on (0 past its end)
__device__ __forceinline__ float4 load4(const float* __restrict__ p, int k, int n, bool vec)
{
    if (vec) return k < n ? __ldg(reinterpret_cast<const float4*>(p + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
    return make_float4(k < n ? __ldg(p + k) : 0.f, k + 1 < n ? __ldg(p + k + 1) : 0.f,
                       k + 2 < n ? __ldg(p + k + 2) : 0.f, k + 3 < n ? __ldg(p + k + 3) : 0.f);
}

__host__ __device__ inline int pad4(int n) { return (n + 3) & ~3; }

// floats of shared memory: input rows, two activation buffers, all pre-activations, the adjoint
// (transposed), the slices of a backward layer
__host__ __device__ inline int rows_smem_floats(const NetDev& p, int R)
{
    int wide = 1, all = 0;
    for (int l = 1; l <= p.L; ++l) {
        wide = wide > p.ld[l] ? wide : p.ld[l];
        all += pad4(p.ld[l]);
    }
    return R * (pad4(p.ld[0]) + 2 * pad4(wide) + all) + pad4(wide) * R + kRowWarps * R * 128;
}

// T values per lane -> the warp's sums, lane l ending with value l (T <= 32, a power of two; shared by
// the 32 / T lanes of equal l / (32 / T) when T < 32)
template <int T>
__device__ __forceinline__ float warp_scatter(float (&v)[T], int lane)
{
    int len = T;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        if (len > 1) {
            const bool up = (lane & o) != 0;
            len >>= 1;
#pragma unroll
            for (int k = 0; k < T / 2; ++k)
                if (k < len) {
                    const float send = up ? v[k] : v[k + len], keep = up ? v[k + len] : v[k];
                    v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    return v[0];
}

template <int R>
__global__ void __launch_bounds__(kRowThreads)
k_mlp_rows(NetDev p, const float* __restrict__ theta, const int32_t* __restrict__ seg_off, const float* __restrict__ G,
           float* __restrict__ E_rows, float* __restrict__ g, int keep)
{
    extern __shared__ float4 sm4[];
    // the CTA's species and rows
    int s = 0, tile = blockIdx.x;
    for (; s < p.S; ++s) {
        const int t = (seg_off[s + 1] - seg_off[s] + R - 1) / R;
        if (tile < t) break;
        tile -= t;
    }
    if (s == p.S) return;
    const int r0 = seg_off[s] + tile * R, nr = min(R, seg_off[s + 1] - r0);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    int wide = 1;
    for (int l = 1; l <= p.L; ++l) wide = max(wide, p.ld[l]);
    float* a0 = reinterpret_cast<float*>(sm4);
    const int lda0 = pad4(p.ld[0]), ldw = pad4(wide);
    float* act[2] = {a0 + R * lda0, a0 + R * (lda0 + ldw)};
    float* zs = act[1] + R * ldw;
    int zoff[kMaxLayers + 2];
    zoff[1] = 0;
    for (int l = 1; l <= p.L; ++l) zoff[l + 1] = zoff[l] + R * pad4(p.ld[l]);
    float* zb = zs + zoff[p.L + 1];          // [unit][row]
    float* slice = zb + ldw * R;
    {
        const int D = p.widths[s][0];
        for (int idx = tid; idx < R * lda0; idx += kRowThreads) {
            const int r = idx / lda0, k = idx - r * lda0;
            a0[idx] = (r < nr && k < D) ? G[(size_t)(r0 + r) * p.ld[0] + k] : 0.f;
        }
    }
    __syncthreads();
    // forward
    const float* in = a0;
    int ldi = lda0;
    for (int l = 0; l < p.L; ++l) {
        const int K = p.widths[s][l], N = p.widths[s][l + 1], at = p.acts[s][l];
        const float* W = theta + p.w_off[s][l];
        const float* bias = theta + p.b_off[s][l];
        const bool vec = (K & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
        float* z = zs + zoff[l + 1];
        const int ldz = pad4(p.ld[l + 1]);
        float* out = act[l & 1];
        for (int n0 = warp * 4; n0 < N; n0 += kRowWarps * 4) {
            float acc[4 * R];
#pragma unroll
            for (int k = 0; k < 4 * R; ++k) acc[k] = 0.f;
#pragma unroll 2
            for (int k = lane * 4; k < K; k += 128) {
                float4 wv[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    wv[j] = n0 + j < N ? load4(W + (size_t)(n0 + j) * K, k, K, vec) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const float4 x = *reinterpret_cast<const float4*>(in + r * ldi + k);
#pragma unroll
                    for (int j = 0; j < 4; ++j)
                        acc[j * R + r] = fmaf(wv[j].x, x.x, fmaf(wv[j].y, x.y, fmaf(wv[j].z, x.z,
                                              fmaf(wv[j].w, x.w, acc[j * R + r]))));
                }
            }
            const float v = warp_scatter<4 * R>(acc, lane);
            constexpr int share = 32 / (4 * R);
            const int e = lane / share, n = n0 + e / R, r = e % R;
            if (lane % share == 0 && n < N) {
                const float zv = v + bias[n], av = act_f(at, zv);
                z[r * ldz + n] = zv;
                out[r * ldw + n] = av;
                if (r < nr) {
                    if (keep) {
                        p.Z[l + 1][(size_t)(r0 + r) * p.ld[l + 1] + n] = zv;
                        p.A[l + 1][(size_t)(r0 + r) * p.ld[l + 1] + n] = av;
                    }
                    if (l == p.L - 1 && n == 0) E_rows[r0 + r] = av;
                }
            }
        }
        // the next layer reads whole groups of four inputs
        if (tid < R)
            for (int n = N; n < pad4(N); ++n) out[tid * ldw + n] = 0.f;
        __syncthreads();
        in = out;
        ldi = ldw;
    }
    if (!g) return;
    // backward: seed dE/da_L = 1
    {
        const int N = p.widths[s][p.L], at = p.acts[s][p.L - 1];
        const float* z = zs + zoff[p.L];
        const int ldz = pad4(p.ld[p.L]);
        for (int idx = tid; idx < N * R; idx += kRowThreads)
            zb[idx] = idx / R == 0 ? act_d1(at, z[(idx % R) * ldz + idx / R]) : 0.f;
    }
    __syncthreads();
    for (int l = p.L - 1; l >= 0; --l) {
        const int K = p.widths[s][l], N = p.widths[s][l + 1];
        const float* W = theta + p.w_off[s][l];
        const bool vec = (K & 3) == 0 && (reinterpret_cast<uintptr_t>(W) & 15) == 0;
        const int kb = (K + 127) / 128, ns = kb < kRowWarps ? kRowWarps / kb : 1;
        const float* z = l > 0 ? zs + zoff[l] : nullptr;
        const int ldz = pad4(p.ld[l]), at = l > 0 ? p.acts[s][l - 1] : 0;
        // kb blocks of 128 inputs at a time while there is a warp for each, all slices side by side
        for (int b0 = 0; b0 < kb; b0 += kRowWarps) {
            const int nb = min(kb - b0, kRowWarps);
            const int blk = warp % nb, sl = warp / nb, k = (b0 + blk) * 128 + lane * 4;
            if (sl < ns) {
                const int n1 = (int)((int64_t)N * (sl + 1) / ns);
                float4 acc[R];
#pragma unroll
                for (int r = 0; r < R; ++r) acc[r] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
                for (int n = (int)((int64_t)N * sl / ns); n < n1; ++n) {
                    const float4 wv = load4(W + (size_t)n * K, k, K, vec);
#pragma unroll
                    for (int r = 0; r < R; r += 4) {
                        const float4 x = *reinterpret_cast<const float4*>(zb + n * R + r);
                        const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            acc[r + q].x = fmaf(xs[q], wv.x, acc[r + q].x);
                            acc[r + q].y = fmaf(xs[q], wv.y, acc[r + q].y);
                            acc[r + q].z = fmaf(xs[q], wv.z, acc[r + q].z);
                            acc[r + q].w = fmaf(xs[q], wv.w, acc[r + q].w);
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r)
                    *reinterpret_cast<float4*>(slice + (size_t)((sl * nb + blk) * R + r) * 128 + lane * 4) = acc[r];
            }
            __syncthreads();
            for (int idx = tid; idx < nb * R * 128; idx += kRowThreads) {
                const int c = idx & 127, r = (idx >> 7) % R, b = (idx >> 7) / R;
                const int kk = (b0 + b) * 128 + c;
                if (kk >= K) continue;
                float v = 0.f;
                for (int q = 0; q < ns && q * nb < kRowWarps; ++q) v += slice[(size_t)((q * nb + b) * R + r) * 128 + c];
                if (l > 0) zb[kk * R + r] = v * act_d1(at, z[r * ldz + kk]);
                else if (r < nr) g[(size_t)(r0 + r) * p.ld[0] + kk] = v;
            }
            __syncthreads();
        }
    }
}

template <int R>
cudaError_t run_rows(const NetDev& p, const float* theta, int64_t N, const int32_t* seg_off, const float* G,
                     float* E_rows, float* g, int keep, size_t smem, cudaStream_t s)
{
    cudaError_t e = allow_smem(k_mlp_rows<R>, smem);
    if (e != cudaSuccess) return e;
    k_mlp_rows<R><<<(unsigned)((N + R - 1) / R + p.S), kRowThreads, smem, s>>>(p, theta, seg_off, G, E_rows, g, keep);
    return cudaGetLastError();
}

}  // namespace

cudaError_t mlp_small_rows(const MlpPlan& p, const MlpBuffers& b, const float* theta, int64_t N, float* E_rows,
                           float* g, bool keep, cudaStream_t s, int* launches)
{
    if (N == 0 || N > kSmallBatch || p.n_out != 1) return cudaErrorNotSupported;
    NetDev d{};
    d.S = p.S; d.L = p.L;
    for (int l = 0; l <= p.L; ++l) {
        d.ld[l] = p.ld[l];
        d.Z[l] = l ? b.Z[l] : nullptr;
        d.A[l] = l ? b.A[l] : nullptr;
    }
    for (int q = 0; q < p.S; ++q)
        for (int l = 0; l <= p.L; ++l) {
            d.widths[q][l] = p.widths[q][l];
            if (l == p.L) break;
            d.acts[q][l] = p.acts[q][l];
            d.w_off[q][l] = p.w_off[q][l];
            d.b_off[q][l] = p.b_off[q][l];
        }
    const int R = N <= 512 ? 4 : 8;
    const size_t smem = (size_t)rows_smem_floats(d, R) * sizeof(float);
    if (smem > 200 * 1024) return cudaErrorNotSupported;
    const cudaError_t e = R == 4 ? run_rows<4>(d, theta, N, b.seg_off, b.G, E_rows, g, keep, smem, s)
                                 : run_rows<8>(d, theta, N, b.seg_off, b.G, E_rows, g, keep, smem, s);
    if (e == cudaSuccess) ++*launches;
    return e;
}

}  // namespace panna
