// Standard Behler-Parrinello angular term: descriptor, adjoint and JVP.
//
// Pair of entries (k1, k2) with vectors a = r_k1, b = r_k2, c = cos(theta), r12 = |b - a| < rc:
//   T_mn = A_m(c) B_n(S) F3,  A_m = 2^(1-zeta_m) (1 + lambda_m c)^zeta_m (0 where 1 + lambda c <= 0),
//   B_n = exp(-eta_n S), S = |a|^2 + |b|^2 + r12^2, F3 = f_c(|a|) f_c(|b|) f_c(r12);
//   dS/da = 4a - 2b, dS/db = 4b - 2a, dc/da = b/(r1 r2) - c a/r1^2, dr12/da = (a - b)/r12,
// plain FP32.  One kernel template for the three uses; a warp per atom, pairs by species block.
//
// Only pairs whose third side is inside the cutoff contribute, about a third of them (two points of a
// ball lie within its radius with probability 0.34).  A warp tests 32 pairs at a time on |b - a|^2
// alone and queues those that pass; the terms themselves run on full rounds of 32 from the queue.
// The tile of (sector, shell) products has the descriptor's size rounded up (4 x 2 to 8 x 8) rather
// than always 8 x 8.  4,096-atom water box, 4 sectors x 2 shells: descriptor 0.55 -> 0.13 ms, adjoint
// 1.47 -> 0.23 ms.
#include <algorithm>

#include "angular.cuh"
#include "common.cuh"

namespace panna {

namespace {

constexpr int kBWarps = 4;
constexpr int kQueue = 64;   // pairs that passed the test and wait: fewer than 32, plus one round
enum { BP_DESC = 0, BP_ADJ = 1, BP_JVP = 2 };

// cos^2(pi x/2) and (pi/2) sin(pi x) for x in [0, 1): f_c and -rc f_c'.  Taylor series of sin and cos
// on [0, pi/4], reflected at x = 1/2, so that both keep their relative accuracy towards x = 1
__device__ __forceinline__ void cutoff_xi(float x, float& f, float& df)
{
    const bool up = x > 0.5f;
    const float t = (up ? 1.f - x : x) * 1.5707963267948966f, t2 = t * t;
    const float s = t * fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, 2.7557319e-6f, -1.9841270e-4f), 8.3333333e-3f),
                                      -0.16666667f), 1.f);
    const float c = fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, fmaf(t2, -2.7557319e-7f, 2.4801587e-5f), -1.3888889e-3f),
                                           4.1666667e-2f), -0.5f), 1.f);
    const float cs = up ? s : c;
    f = cs * cs;
    df = 3.14159265358979f * s * c;
}

// A_m and dA_m/dc of the sectors from m0 on
template <int TM, bool SLOPE>
__device__ __forceinline__ void bp_sectors(const DescDev& d, int m0, float c, float (&A)[TM], float (&dA)[TM])
{
#pragma unroll
    for (int k = 0; k < TM; ++k) {
        const int m = min(m0 + k, d.n_theta - 1);
        const float lam = d.bp_lambda[m];
        const float y = fmaxf(fmaf(lam, c, 1.f), 0.f);
        const int zi = d.bp_zeta_int[m];
        float p1;   // y^(zeta - 1)
        if (zi > 0) {
            p1 = 1.f;
            float base = y;
            for (int e = zi - 1; e; e >>= 1) {
                if (e & 1) p1 *= base;
                base *= base;
            }
        } else {
            p1 = ex2f((d.bp_zeta[m] - 1.f) * lg2f(fmaxf(y, 1e-37f)));
        }
        if (SLOPE) dA[k] = y > 0.f ? d.bp_pref[m] * d.bp_zeta[m] * lam * p1 : 0.f;
        A[k] = d.bp_pref[m] * p1 * y;
    }
}

__host__ __device__ inline int bp_warp_floats(int cap, int mode, int nc)
{
    return cap * 8 + (mode == BP_ADJ ? 4 * nc * cap : mode == BP_JVP ? 4 * cap : 0) + 2 * kQueue;
}

template <int MODE, int TM, int TN>
__global__ void __launch_bounds__(kBWarps * 32)
k_bp(DescDev d, Work w, const int32_t* __restrict__ row_map, const float* __restrict__ in, float* __restrict__ out,
     float* __restrict__ F, float* __restrict__ vir_atom, int nc)
{
    extern __shared__ float4 sm4[];
    __shared__ int s_seg[kBWarps][kMaxSpecies + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cap = w.cap;
    float* base = reinterpret_cast<float*>(sm4) + (size_t)warp * bp_warp_floats(cap, MODE, nc);
    float4* sv = reinterpret_cast<float4*>(base);   // (v, r)
    float4* sx = sv + cap;                          // (1/r, f_c, f_c', JVP: dr/dt)
    float4* sq = sx + cap;                          // adjoint: nc copies of the entry sums; JVP: tangents
    int2* queue = reinterpret_cast<int2*>(sq + (MODE == BP_ADJ ? nc * cap : MODE == BP_JVP ? cap : 0));
    int* seg = s_seg[warp];
    const int nbins = d.n_theta * d.n_ang_r;
    const float inv_rc = 1.f / d.rc;
    for (int64_t i = (int64_t)blockIdx.x * kBWarps + warp; i < w.N; i += (int64_t)gridDim.x * kBWarps) {
        const int64_t row = row_map ? row_map[i] : i;
        if (row < 0) continue;   // ghosts are not centres
        const int n = w.nb_count[i];
        const size_t sb = (size_t)i * cap;
        const float* gi = MODE == BP_ADJ ? in + (size_t)row * d.D : nullptr;
        float* Oi = MODE != BP_ADJ ? out + (size_t)row * d.D : nullptr;
        __syncwarp();   // the previous atom's reads of the staging area are done
        float uix = 0.f, uiy = 0.f, uiz = 0.f;
        if (MODE == BP_JVP) { uix = in[3 * i]; uiy = in[3 * i + 1]; uiz = in[3 * i + 2]; }
        for (int k = lane; k < n; k += 32) {
            const float4 v = w.nb_vec[sb + k];
            const float ir = 1.f / v.w;
            sv[k] = v;
            float s_, c_, rd = 0.f;
            sincospif(0.5f * (v.w / d.rc), &s_, &c_);
            if (MODE == BP_JVP) {
                const int64_t j = w.nb_idx[sb + k].x;
                const float a = in[3 * j] - uix, b = in[3 * j + 1] - uiy, c = in[3 * j + 2] - uiz;
                rd = fmaf(v.x, a, fmaf(v.y, b, v.z * c)) * ir;
                sq[k] = make_float4(a, b, c, 0.f);
            }
            sx[k] = make_float4(ir, c_ * c_, -d.pi_rc * s_ * c_, rd);
            if (MODE == BP_ADJ)
                for (int c = 0; c < nc; ++c) sq[c * cap + k] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        species_segments(d, w.nb_idx + sb, n, seg, lane);
        __syncwarp();

        // radial terms
        if (MODE == BP_ADJ) {
            // sum_n g_n d/dr of the entry's shells, as the coefficient of its own vector
            for (int k = lane; k < n; k += 32) {
                int s = 0;
                while (k >= seg[s + 1]) ++s;
                const float* gr = gi + s * d.n_rad;
                const float r = sv[k].w, fc = sx[k].y, dfc = sx[k].z;
                float T = 0.f;
                for (int nn = 0; nn < d.n_rad; ++nn) {
                    const float x = r - d.rs_rad[nn];
                    T = fmaf(gr[nn] * __expf(-d.eta_rad * x * x), fmaf(-2.f * d.eta_rad * x, fc, dfc), T);
                }
                sq[k].w = T * sx[k].x;
            }
        } else {
            for (int nn = lane; nn < d.n_rad; nn += 32) {
                const float rs = d.rs_rad[nn];
                for (int s = 0; s < d.S; ++s) {
                    float acc = 0.f;
                    for (int k = seg[s]; k < seg[s + 1]; ++k) {
                        const float x = sv[k].w - rs;
                        const float e = __expf(-d.eta_rad * x * x);
                        acc = MODE == BP_DESC ? fmaf(e, sx[k].y, acc)
                                              : fmaf(e * fmaf(-2.f * d.eta_rad * x, sx[k].y, sx[k].z), sx[k].w, acc);
                    }
                    Oi[s * d.n_rad + nn] = acc;
                }
            }
        }
        __syncwarp();

        for (int m0 = 0; m0 < d.n_theta; m0 += TM)
        for (int n0 = 0; n0 < d.n_ang_r; n0 += TN) {
            float eta[TN];
#pragma unroll
            for (int k = 0; k < TN; ++k) eta[k] = d.bp_eta[min(n0 + k, d.n_ang_r - 1)];
            int blk = 0;
            for (int a = 0; a < d.S; ++a)
            for (int b = a; b < d.S; ++b, ++blk) {
                BlockPairs bp(seg[a], seg[a + 1] - seg[a], seg[b], seg[b + 1] - seg[b], a == b, lane);
                float gv[MODE == BP_ADJ ? TM : 1][TN];
                float acc[MODE == BP_ADJ ? 1 : TM * TN];
                if (MODE == BP_ADJ) {
                    if (bp.n == 0) continue;
                    const float* gb = gi + d.rad_cols + blk * nbins;
#pragma unroll
                    for (int mm = 0; mm < TM; ++mm)
#pragma unroll
                        for (int q = 0; q < TN; ++q) {
                            const int m = m0 + mm, nq = n0 + q;
                            gv[MODE == BP_ADJ ? mm : 0][q] =
                                (m < d.n_theta && nq < d.n_ang_r) ? gb[m * d.n_ang_r + nq] : 0.f;
                        }
                } else {
#pragma unroll
                    for (int k = 0; k < (MODE == BP_ADJ ? 1 : TM * TN); ++k) acc[k] = 0.f;
                }
                // the terms of the queue's first `cnt` pairs, one per lane
                auto process = [&](int head, int cnt) {
                    const bool on = lane < cnt;
                    const int2 e = queue[(head + (on ? lane : 0)) & (kQueue - 1)];
                    const int k1 = e.x & 0xffff, k2 = e.x >> 16;
                    const float4 va = sv[k1], vb = sv[k2], xa = sx[k1], xb = sx[k2];
                    const float dx = vb.x - va.x, dy = vb.y - va.y, dz = vb.z - va.z;
                    const float r12s = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                    const float r12 = sqrt_nr(r12s), i12 = MODE != BP_DESC && r12 > 0.f ? rcpf(r12) : 0.f;
                    float f12, d12;
                    const float xi = r12 * inv_rc;
                    cutoff_xi(fmaf(inv_rc, fmaf(-d.rc, xi, r12), xi), f12, d12);
                    d12 *= -inv_rc;   // f_c'(r12)
                    const float ir12 = xa.x * xb.x;
                    const float c = fmaf(va.x, vb.x, fmaf(va.y, vb.y, va.z * vb.z)) * ir12;
                    const float f11 = xa.y * xb.y;
                    const float F3 = on ? f11 * f12 : 0.f;
                    const float S = fmaf(va.w, va.w, fmaf(vb.w, vb.w, r12s));
                    float A[TM], dA[TM], B[TN];
                    bp_sectors<TM, MODE != BP_DESC>(d, m0, c, A, dA);
#pragma unroll
                    for (int q = 0; q < TN; ++q) B[q] = __expf(-eta[q] * S);
                    if (MODE == BP_DESC) {
#pragma unroll
                        for (int mm = 0; mm < TM; ++mm)
#pragma unroll
                            for (int q = 0; q < TN; ++q)
                                acc[MODE == BP_DESC ? mm * TN + q : 0] = fmaf(A[mm] * F3, B[q],
                                                                              acc[MODE == BP_DESC ? mm * TN + q : 0]);
                    } else if (MODE == BP_JVP) {
                        // tangents of c, S and F3 along (v_k1, v_k2)
                        const float4 t1 = sq[k1], t2 = sq[k2];
                        const float a1 = xa.w * va.w, b2 = xb.w * vb.w;   // a . t1, b . t2
                        const float b1 = fmaf(vb.x, t1.x, fmaf(vb.y, t1.y, vb.z * t1.z));
                        const float a2 = fmaf(va.x, t2.x, fmaf(va.y, t2.y, va.z * t2.z));
                        const float cd = fmaf(-c * xa.x, xa.w, b1 * ir12) + fmaf(-c * xb.x, xb.w, a2 * ir12);
                        const float sd = 4.f * (a1 + b2) - 2.f * (b1 + a2);
                        const float abv = (dx * (t2.x - t1.x) + dy * (t2.y - t1.y) + dz * (t2.z - t1.z)) * i12;
                        const float Fd = on ? f12 * fmaf(xa.z * xa.w, xb.y, xa.y * xb.z * xb.w) + f11 * d12 * abv : 0.f;
                        const float Fc = F3 * cd;
#pragma unroll
                        for (int q = 0; q < TN; ++q) {
                            const float H = fmaf(-eta[q] * sd, F3, Fd);
#pragma unroll
                            for (int mm = 0; mm < TM; ++mm)
                                acc[MODE == BP_JVP ? mm * TN + q : 0] =
                                    fmaf(B[q], fmaf(dA[mm], Fc, A[mm] * H), acc[MODE == BP_JVP ? mm * TN + q : 0]);
                        }
                    } else {
                        float Tc = 0.f, TS = 0.f, TF = 0.f;
#pragma unroll
                        for (int q = 0; q < TN; ++q) {
                            float ga = 0.f, gd = 0.f;
#pragma unroll
                            for (int mm = 0; mm < TM; ++mm) {
                                ga = fmaf(gv[MODE == BP_ADJ ? mm : 0][q], A[mm], ga);
                                gd = fmaf(gv[MODE == BP_ADJ ? mm : 0][q], dA[mm], gd);
                            }
                            Tc = fmaf(gd, B[q], Tc);
                            TF = fmaf(ga, B[q], TF);
                            TS = fmaf(-eta[q] * ga, B[q], TS);
                        }
                        Tc *= F3;
                        TS *= F3;
                        // gradient on entry 1 = al1 a + be b, on entry 2 = al2 b + be a: entry sums hold
                        // the other entries' vectors and the coefficient of the own one
                        const float T12 = TF * f11 * d12 * i12;
                        const float be = fmaf(Tc, ir12, -2.f * TS) - T12;
                        const float al1 = fmaf(-Tc * c, xa.x * xa.x, 4.f * TS) + fmaf(TF * xa.z * xb.y * f12, xa.x, T12);
                        const float al2 = fmaf(-Tc * c, xb.x * xb.x, 4.f * TS) + fmaf(TF * xa.y * xb.z * f12, xb.x, T12);
                        const int q0 = __shfl_sync(0xffffffffu, e.y, 0);
                        const int nd = __shfl_sync(0xffffffffu, e.y, cnt - 1) - q0 + 1, qd = e.y - q0;
                        // the entries of one diagonal are distinct; its sums go to their own copy
                        for (int c0 = 0; c0 < nd; c0 += nc) {
                            const bool act = on && qd >= c0 && qd < c0 + nc;
                            if (!__any_sync(0xffffffffu, act)) continue;
                            float4* cp = sq + (qd - c0) * cap;
                            if (act) {
                                const float4 o = cp[k1];
                                cp[k1] = make_float4(fmaf(be, vb.x, o.x), fmaf(be, vb.y, o.y), fmaf(be, vb.z, o.z),
                                                     o.w + al1);
                            }
                            __syncwarp();
                            if (act) {
                                const float4 o = cp[k2];
                                cp[k2] = make_float4(fmaf(be, va.x, o.x), fmaf(be, va.y, o.y), fmaf(be, va.z, o.z),
                                                     o.w + al2);
                            }
                            __syncwarp();
                        }
                    }
                };
                int head = 0, cnt = 0;
                for (int p0 = 0; p0 < bp.n; p0 += 32, bp.next()) {
                    bool on = p0 + lane < bp.n;
                    int k1, k2;
                    bp.get(on, k1, k2);
                    const float4 va = sv[k1], vb = sv[k2];
                    const float dx = vb.x - va.x, dy = vb.y - va.y, dz = vb.z - va.z;
                    on = on && fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < d.rc2;
                    const unsigned hit = __ballot_sync(0xffffffffu, on);
                    if (on)
                        queue[(head + cnt + __popc(hit & ((1u << lane) - 1u))) & (kQueue - 1)] =
                            make_int2(k1 | (k2 << 16), bp.q);
                    cnt += __popc(hit);
                    __syncwarp();
                    if (cnt >= 32) {
                        process(head, 32);
                        head = (head + 32) & (kQueue - 1);
                        cnt -= 32;
                        __syncwarp();
                    }
                }
                if (cnt > 0) process(head, cnt);
                __syncwarp();
                if (MODE != BP_ADJ) {
                    // sums over the lanes in a fixed order; lane l ends with element l / (32 / (TM TN))
                    constexpr int T = TM * TN;
                    float v[MODE == BP_ADJ ? 1 : T];
#pragma unroll
                    for (int k = 0; k < (MODE == BP_ADJ ? 1 : T); ++k) v[k] = acc[k];
                    int len = T;
#pragma unroll
                    for (int o = 16; o >= 1; o >>= 1) {
                        if (len > 1) {
                            const bool up = (lane & o) != 0;
                            len >>= 1;
#pragma unroll
                            for (int k = 0; k < T / 2; ++k) {
                                if (k < len && MODE != BP_ADJ) {
                                    const float send = up ? v[MODE == BP_ADJ ? 0 : k] : v[MODE == BP_ADJ ? 0 : k + len];
                                    const float keep = up ? v[MODE == BP_ADJ ? 0 : k + len] : v[MODE == BP_ADJ ? 0 : k];
                                    v[MODE == BP_ADJ ? 0 : k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                                }
                            }
                        } else {
                            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
                        }
                    }
                    constexpr int per = T >= 32 ? T / 32 : 1;        // elements a lane ends with
                    constexpr int share = T >= 32 ? 1 : 32 / T;      // lanes that end with the same one
                    float* Ob = Oi + d.rad_cols + blk * nbins;
                    if (lane % share == 0) {
#pragma unroll
                        for (int k = 0; k < per; ++k) {
                            const int e = lane / share * per + k;
                            const int m = m0 + e / TN, q = n0 + e % TN;
                            if (m < d.n_theta && q < d.n_ang_r) Ob[m * d.n_ang_r + q] = v[MODE == BP_ADJ ? 0 : k];
                        }
                    }
                }
            }
        }
        if (MODE == BP_ADJ) {
            __syncwarp();
            float fx = 0.f, fy = 0.f, fz = 0.f, vv[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) vv[k] = 0.f;
            for (int k = lane; k < n; k += 32) {
                float4 z = sq[k];
                for (int c = 1; c < nc; ++c) {
                    const float4 o = sq[c * cap + k];
                    z.x += o.x; z.y += o.y; z.z += o.z; z.w += o.w;
                }
                const float4 v = sv[k];
                const float q[3] = {fmaf(z.w, v.x, z.x), fmaf(z.w, v.y, z.y), fmaf(z.w, v.z, z.z)};
                fx += q[0]; fy += q[1]; fz += q[2];
                const int64_t j = w.nb_idx[sb + k].x;
                atomicAdd(&F[3 * j + 0], -q[0]);
                atomicAdd(&F[3 * j + 1], -q[1]);
                atomicAdd(&F[3 * j + 2], -q[2]);
                const float rv[3] = {v.x, v.y, v.z};
#pragma unroll
                for (int aa = 0; aa < 3; ++aa)
#pragma unroll
                    for (int bb = 0; bb < 3; ++bb) vv[3 * aa + bb] -= q[aa] * rv[bb];
            }
            add_centre(w, i, fx, fy, fz, vv, F, vir_atom, lane);
        }
    }
}

}  // namespace

template <int MODE>
cudaError_t launch_bp(const Work& w, const DescDev& d, const int32_t* row_map, const float* in, float* out, float* F,
                      float* vir_atom, cudaStream_t s, int* launches)
{
    if (w.N == 0) return cudaSuccess;
    int nc = MODE == BP_ADJ ? 4 : 1;
    while (nc > 1 && (size_t)kBWarps * bp_warp_floats(w.cap, MODE, nc) * 4 > 40 * 1024) nc /= 2;
    const size_t smem = (size_t)kBWarps * bp_warp_floats(w.cap, MODE, nc) * 4;
    auto run = [&](auto kern) {
        cudaError_t e = allow_smem(kern, smem);
        if (e != cudaSuccess) return e;
        kern<<<(unsigned)((w.N + kBWarps - 1) / kBWarps), kBWarps * 32, smem, s>>>(d, w, row_map, in, out, F, vir_atom,
                                                                                  nc);
        ++*launches;
        return cudaGetLastError();
    };
    // the smallest tile that holds all (sector, shell) products; larger sets take several passes
    if (d.n_theta <= 4 && d.n_ang_r <= 2) return run(k_bp<MODE, 4, 2>);
    if (d.n_theta <= 4 && d.n_ang_r <= 4) return run(k_bp<MODE, 4, 4>);
    if (d.n_ang_r <= 4) return run(k_bp<MODE, 8, 4>);
    return run(k_bp<MODE, 8, 8>);
}

template cudaError_t launch_bp<0>(const Work&, const DescDev&, const int32_t*, const float*, float*, float*, float*,
                                  cudaStream_t, int*);
template cudaError_t launch_bp<1>(const Work&, const DescDev&, const int32_t*, const float*, float*, float*, float*,
                                  cudaStream_t, int*);
template cudaError_t launch_bp<2>(const Work&, const DescDev&, const int32_t*, const float*, float*, float*, float*,
                                  cudaStream_t, int*);

}  // namespace panna
