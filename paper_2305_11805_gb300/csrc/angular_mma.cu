// Angular descriptor, its adjoint and its tangent with the products over sectors and shells on the warp-level
// tensor cores (modified angular term; the forms are those of descriptor.cu).
//
// What is different from the one-lane-per-pair kernels.  Per pair of neighbours the angular term
// is an outer product A (x) e of n_theta sector powers and n_R shell Gaussians.  A lane that owns a
// pair evaluates 8 + 8 of them, reads the sectors' and shells' constants from shared memory for
// each, and holds (descriptor) a 64-float tile or reads (adjoint) a 64-float tile per pair.  Here a
// warp takes its pairs 32 at a time in two steps.  Step 1, a lane per pair: the geometry (half
// angles, mean distance), left in shared memory.  Step 2, lanes in the layout of the MMA operands:
// lane (g, t) = (lane / 4, lane mod 4) evaluates sector g and shell g for pairs t, t + 4 of each
// group of 8, so the sector's and shell's constants stay in its registers, two pairs share every
// two-wide FP32 instruction, and mma.m16n8k8 contracts over the pairs.  The tile is 4 registers.
// (The contraction is 8 x 8 x 8 per group of pairs of one atom, far below the 128-row tiles of
// tcgen05, whose operands would have to pass through shared memory besides.)
//
// What bounds it (ncu, water box of 16,384 atoms): instruction issue, two-wide FP32 instructions taking
// two dispatch cycles each, next to the shared-memory data path.  A round of 32 pairs takes about 214
// warp instructions (fast descriptor) against 400 in the lane-per-pair kernel; mma.m16n8k8 with TF32
// operands issues every 8 cycles per scheduler and is 20 % busy.  Pair buffers hold what a
// lane reads as 4-byte words because a load returns at most 128 bytes a cycle to the warp, also when
// its lanes share addresses.
//
// Measured (GB300, before -> after, ms per launch; before: descriptor.cu's compensated or float-pair
// descriptor and its diagonal-order adjoint):
//                                            BF16 networks                FP32 networks
//                                       descriptor     adjoint       descriptor     adjoint
//   128 ragged boxes (107,202 atoms)   1.03 -> 0.74  1.39 -> 1.20   2.48 -> 1.31  1.66 -> 1.51
//   water box (16,384 atoms)           0.67 -> 0.59  1.26 -> 0.94   1.89 -> 1.16  1.57 -> 1.26
//   FCC box (131,072 atoms)            1.66 -> 1.07  2.56 -> 1.66   4.47 -> 2.3   3.13 -> 2.14
//   1024 molecules (17,396 atoms)      0.14 -> 0.07  0.125 -> 0.117 0.23 -> 0.10  0.145 -> 0.133
// Below zeta = 16 (FP32 networks, 4,096 atoms, 47 neighbours): descriptor 172 (230 with fractional exponents) ->
// 155 us, adjoint 150 -> 125.  The 16-sector descriptors of FP32 networks spill 32 and 40 bytes.
//
// FP32 accuracy on TF32 operands: every operand is split into hi + lo TF32 parts (hi its leading 11
// bits, lo the exact rest), so products carry about 22 bits; the descriptor puts A_hi in rows 0..7
// and A_lo in rows 8..15 of one A operand.  The tensor cores accumulate a round of 32 pairs, which
// is then added to the block's sum in plain FP32.
//
// The eps-regularised angle.  With R = sqrt(1 + eps), (cos, sin_eps) = R (cos th', sin th') exactly,
// so 1 - y_m = t_m = R sin^2((th' - theta_m)/2) - (R - 1)/2: one angle th' per pair carries eps, and
// sin, cos of (th' - theta_m)/2 come from the half angles of th' with relative accuracy.
//
// Two arithmetics.  FAST (the BF16 networks' rows, 16 significant bits): hardware square roots and
// y^zeta = 2^(zeta log2 y) from the hardware log2 (absolute error 2^-22).  Otherwise Newton steps and
// y^zeta = 2^(zeta log2(1 - t)) from the Taylor series of the logarithm: y^zeta exceeds 2^-30 only for
// small t, and dropping the terms from t^(d+1) on moves y^zeta by at most
// zeta t^(d+1)/(d+1) (1-t)^zeta <= 1.5e-9 (d = 8, zeta >= 32), 1.1e-9 (d = 13, zeta >= 16) of its
// maximum; all terms have one sign, so for t near 1 the sum still underflows as y^zeta does.  Below
// zeta = 16, and where eps makes the series too short, the power comes from the float pair 1 - t.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>

#include "angular.cuh"
#include "common.cuh"

namespace panna {

namespace {

constexpr int kMW = 4;        // warps per CTA, an atom each
constexpr int kTeamMax = 8;   // warps of a CTA that share one atom (TEAM), and
constexpr int kTeamCtas = 8;  // CTAs (a cluster), at most

namespace cg = cooperative_groups;

// TEAM: the part of a warp in the rounds of 32 pairs of one species block.  All blocks' rounds, in order,
// are dealt to the warps in consecutive runs [lo, hi); rb counts the rounds before the block.
struct TeamRounds {
    int R = 0, lo, hi, rb = 0;
    __device__ __forceinline__ TeamRounds(const DescDev& d, const int* seg, int warp, int warps)
    {
        for (int a = 0; a < d.S; ++a)
            for (int b = a; b < d.S; ++b) R += rounds(block_pairs(seg, a, b));
        lo = R * warp / warps;
        hi = R * (warp + 1) / warps;
    }
    static __device__ __forceinline__ int block_pairs(const int* seg, int a, int b)
    {
        const int na = seg[a + 1] - seg[a];
        return a == b ? na * (na - 1) / 2 : na * (seg[b + 1] - seg[b]);
    }
    static __device__ __forceinline__ int rounds(int pairs) { return (pairs + 31) / 32; }
    // the warp's rounds [first, last) of the next block
    __device__ __forceinline__ void next(int pairs, int& first, int& last)
    {
        const int nr = rounds(pairs);
        first = max(lo - rb, 0);
        last = min(hi - rb, nr);
        rb += nr;
    }
};

// D += A B, m16n8k8, TF32 operands (the leading 19 bits of each register), FP32 accumulators
__device__ __forceinline__ void mma8(float (&c)[4], float a0, float a1, float a2, float a3, float b0, float b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(__float_as_uint(a0)), "r"(__float_as_uint(a1)), "r"(__float_as_uint(a2)),
                   "r"(__float_as_uint(a3)), "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)));
}

// D = A B
__device__ __forceinline__ void mma8z(float (&c)[4], float a0, float a1, float a2, float a3, float b0, float b1)
{
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                 "{%10,%10,%10,%10};"
                 : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
                 : "r"(__float_as_uint(a0)), "r"(__float_as_uint(a1)), "r"(__float_as_uint(a2)),
                   "r"(__float_as_uint(a3)), "r"(__float_as_uint(b0)), "r"(__float_as_uint(b1)), "f"(0.f));
}

__device__ __forceinline__ float tf_hi(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// x = hi + lo exactly; hi has the bits that TF32 keeps.  ROUND: hi to nearest, so that lo is signed
// and what the tensor cores drop of it (its bits past 11) has no bias.
template <bool ROUND>
__device__ __forceinline__ void tf_split(float2 x, float2& hi, float2& lo)
{
    const uint32_t r = ROUND ? 0x1000u : 0u;
    hi = make_float2(__uint_as_float((__float_as_uint(x.x) + r) & 0xffffe000u),
                     __uint_as_float((__float_as_uint(x.y) + r) & 0xffffe000u));
    lo = __fadd2_rn(x, make_float2(-hi.x, -hi.y));
}

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

// zeta log2(1 - t) (or zeta - 1: coefficients zl) to degree PW, see the file comment
template <int PW>
__device__ __forceinline__ float2 log_series(const float* zl, float2 t)
{
    float2 p = dup(zl[PW - 1]);
#pragma unroll
    for (int k = PW - 2; k >= 0; --k) p = __ffma2_rn(p, t, dup(zl[k]));
    return __fmul2_rn(p, t);
}

// (1 - t)^e below e = 16, from the float pair yh + yl = 1 - t.  LIB: the library's logarithm; the hardware's,
// off by up to 2^-22, made descriptor rows of zeta = 15.5 2.4 times as far off as the blocked kernel's, and
// repeated squaring for whole exponents took 1 to 10 us more of 155 (4,096 atoms, 47 neighbours).  The adjoint's
// forces are bound by the angle in single floats, as those of its other kernels, which take the hardware's too
// (0.95 to 1.03 times the diagonal-order kernel's error with either; 191 us with the library's or with a loop of
// squarings, 125 so).
template <bool LIB>
__device__ __forceinline__ float pow_low(float e, float t)
{
    const float yh = 1.f - t;
    const float yl = (1.f - yh) - t;
    if (!(yh > 0.f)) return 0.f;
    const float z = e * fmaf(yl * rcpf(yh), 1.4426950408889634f, LIB ? log2f(yh) : lg2f(yh));
    return LIB ? exp2f(z) : ex2f(z);
}

// (1 - t)^zeta, zeta the exponent of the coefficients zl
template <int PW, bool LIB>
__device__ __forceinline__ float2 pow2_t(const float* zl, float zeta, float2 t)
{
    if (PW == 0) return make_float2(pow_low<LIB>(zeta, t.x), pow_low<LIB>(zeta, t.y));
    const float2 z = log_series<PW ? PW : 1>(zl, t);
    return make_float2(ex2f(z.x), ex2f(z.y));
}

// y^zeta = 2^(zeta log2 |y|) (FAST): where no_clamp lets it stand for max(y, 0)^zeta
__device__ __forceinline__ float2 pow2_y(float zeta, float2 y)
{
    const float2 z = __fmul2_rn(make_float2(lg2f(fabsf(y.x)), lg2f(fabsf(y.y))), dup(zeta));
    return make_float2(ex2f(z.x), ex2f(z.y));
}

// Half angles (sin, cos of th'/2) from cos(theta) and sin_eps^2(theta): the one of (1 + |cos th'|)/2
// without cancellation by a square root, the other from sin th' / 2
template <bool FAST>
__device__ __forceinline__ void half_angles(const DescDev& d, float c, float se2, float& sh, float& ch)
{
    float hq, o;
    const float q = fmaf(0.5f * d.r_inv, fabsf(c), 0.5f);   // in [1/2, 1]
    if (FAST) {
        const float iq = rsqf(q);
        hq = q * iq;
        o = (0.5f * d.r_inv) * se2 * rsqf(fmaxf(se2, 1e-37f)) * iq;
    } else {
        hq = sqrt_nr(q);
        o = div_nr(0.5f * d.r_inv * sqrt_nr(se2), hq);
    }
    ch = c >= 0.f ? hq : o;
    sh = c >= 0.f ? o : hq;
}

// sqrt((1 + c + cl)/2) as hi + lo, c + cl >= -1
__device__ __forceinline__ void half_pair(float c, float cl, float& h, float& l)
{
    float qh, ql;
    two_sum(1.f, c, qh, ql);
    ql += cl;
    fast_two_sum(qh, ql, qh, ql);   // near c = -1 the low part is a large fraction
    qh = fmaxf(0.5f * qh, 0.f);
    h = sqrt_nr(qh);
    l = h > 0.f ? fmaf(0.5f, ql, fmaf(-h, h, qh)) * (0.5f * rcpf(h)) : 0.f;
}

// ------------------------------------------------------------------ descriptor

// Arithmetic of the descriptor kernel.  FAST: see the file comment.  PAIR (FP32 networks, whose
// forces have to meet 1e-5 of RMS): the half angles as float pairs.  Rounding them to single floats
// moves the angle by about 3e-8, which the zeta-th power turns into 1e-6 of a term.  The error of a
// rounded (sin, cos) along the circle is one angle delta per pair, so that
//   sin((th' - theta_m)/2) = [sh cos_m - ch sin_m] + (delta - delta_m) cos((th' - theta_m)/2),
// the bracket by an FMA-compensated difference of products, delta_m the same error of the sector's
// constants.  Distances enter as the exact sum r1 + r2 = 2 (hi + lo).

// TEAM (small batches): all warps of a cluster of CTAs share one atom and its rounds (TeamRounds), those of
// a CTA its staging area.  The runs are consecutive, so a warp writes the blocks that are wholly its own;
// of a block shared with the warps after it the first warp adds up the others' sums, in order, those of
// the cluster's other CTAs CTA by CTA through distributed shared memory.

// shared bytes of an atom: unit vectors and distances (PAIR: and their low parts), r, f_c
template <bool FAST>
__host__ __device__ inline size_t desc_mma_atom_bytes(int cap)
{
    return FAST ? (size_t)((cap + 1) & ~1) * (16 + 4 + 4) : (size_t)cap * (16 + 16);
}
// and of a warp: the round's pairs (TEAM: and its part of a shared block)
template <bool FAST>
__host__ __device__ inline size_t desc_mma_warp_bytes(int part)
{
    return 16 * (FAST ? 16 + 16 : 16 + 16 + 16) + part * 512;
}

template <bool FAST, int CM, int PW, bool TEAM>
__global__ void __launch_bounds__((TEAM ? kTeamMax : kMW) * 32,
                                  TEAM ? 2 : FAST ? (CM == 1 ? 8 : 7) : (CM == 1 ? 6 : 5))
k_desc_mma(DescDev d, Work w, const int32_t* __restrict__ row_map, float* __restrict__ out,
           __nv_bfloat16* __restrict__ Gh, __nv_bfloat16* __restrict__ Gl, int even)
{
    extern __shared__ float4 sm4[];
    __shared__ int s_seg[TEAM ? kTeamMax : kMW][kMaxSpecies + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cap = w.cap, cap2 = (cap + 1) & ~1;
    const int warps = TEAM ? blockDim.x >> 5 : 1, tid = TEAM ? threadIdx.x : lane, threads = 32 * warps;
    const size_t a_bytes = desc_mma_atom_bytes<FAST>(cap), w_bytes = desc_mma_warp_bytes<FAST>(TEAM ? CM : 0);
    char* base = reinterpret_cast<char*>(sm4) + (TEAM ? 0 : warp * (a_bytes + w_bytes));
    const int ctas = TEAM ? cg::this_cluster().num_blocks() : 1, rank = TEAM ? cg::this_cluster().block_rank() : 0;
    const int wt = rank * warps + warp, team = ctas * warps;   // the warp's number among those of its atom
    auto sync = [] {
        if (TEAM) __syncthreads();
        else __syncwarp();
    };
    auto cluster_sync = [&] {
        if (ctas > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    // FAST: (unit vector, rho = (r - R_c) sqrt(eta_l) / 2), r, f_c; PAIR: (unit vector, r), (its low
    // part, f_c).  rho: distances relative to the middle shell R_c in units of the Gaussians' width, so
    // that exp(-eta (r_bar - R)^2) = 2^(-x^2) with x = rho_1 + rho_2 - (R - R_c) sqrt(eta_l); rounding
    // r - R_c instead of r keeps the small x of the terms that count
    float4* sv = reinterpret_cast<float4*>(base);
    float4* sl = sv + cap;
    float* sr = reinterpret_cast<float*>(sv + cap2);
    float* sf = sr + cap2;
    const float r_c = d.rs_ang[d.n_ang_r / 2], s_eta = sqrtf(d.eta_ang * 1.4426950408889634f);
    // geometry of the round's pairs, each for pairs t and t + 4 of a group.  pa: sin, cos of th'/2;
    // pr: FAST x + nR, f_c f_c; PAIR: the halves of r_bar; pd: PAIR delta, f_c f_c.  Groups 2 and 3
    // swap the two halves of each float4, so that the 32 lanes' stores fall on 32 banks
    float4* pa = reinterpret_cast<float4*>(base + a_bytes + (TEAM ? warp * w_bytes : 0));
    float4* pr = pa + 16;
    float4* pd = pr + 16;
    float4* part = pd + 16;   // TEAM: [CM][32] accumulators of a block begun by a warp before this one
    // this lane's slot of the pair buffers when it owns pair `lane`
    const int slot = (lane >> 3) * 4 + t, half = (lane >> 2) & 1;
    const int off0 = slot * 4 + half + ((lane >> 4) << 1), off1 = slot * 4 + half + (2 - ((lane >> 4) << 1));
    float* pa_f = reinterpret_cast<float*>(pa);
    float* pr_f = reinterpret_cast<float*>(pr);
    float* pd_f = reinterpret_cast<float*>(pd);
    int* seg = s_seg[warp];
    const int ncm = (d.n_theta + 7) / 8, ncn = (d.n_ang_r + 7) / 8;
    const int nbins = d.n_theta * d.n_ang_r;
    const float eta_rl = d.eta_rad * 1.4426950408889634f;   // exp(-eta x^2) = 2^(-eta_l x^2)
    auto put = [&](size_t idx, float v) {
        if (Gh) {
            const __nv_bfloat16 h = __float2bfloat16_rn(v);
            Gh[idx] = h;
            if (Gl) Gl[idx] = __float2bfloat16_rn(v - __bfloat162float(h));
        } else {
            out[idx] = v;
        }
    };
    auto put2 = [&](size_t idx, float v0, float v1) {
        if (Gh) {
            const __nv_bfloat16 h0 = __float2bfloat16_rn(v0), h1 = __float2bfloat16_rn(v1);
            *reinterpret_cast<__nv_bfloat162*>(Gh + idx) = __nv_bfloat162(h0, h1);
            if (Gl)
                *reinterpret_cast<__nv_bfloat162*>(Gl + idx) =
                    __nv_bfloat162(__float2bfloat16_rn(v0 - __bfloat162float(h0)),
                                   __float2bfloat16_rn(v1 - __bfloat162float(h1)));
        } else {
            *reinterpret_cast<float2*>(out + idx) = make_float2(v0, v1);
        }
    };
    for (int64_t i = TEAM ? blockIdx.x / ctas : (int64_t)blockIdx.x * kMW + warp; i < w.N;
         i += TEAM ? gridDim.x / ctas : (int64_t)gridDim.x * kMW) {
        const int64_t row = row_map ? row_map[i] : i;
        if (row < 0) continue;   // ghosts are not centres
        const int n = w.nb_count[i];
        const size_t sb = (size_t)i * cap;
        sync();   // the previous atom's reads of the staging area are done
        for (int k = tid; k < n; k += threads) {
            const float4 v = w.nb_vec[sb + k];
            if (FAST) {
                const float ir = 1.f / v.w;
                sv[k] = make_float4(v.x * ir, v.y * ir, v.z * ir, (v.w - r_c) * (0.5f * s_eta));
                const float c_ = cospif(0.5f * (v.w / d.rc));
                sr[k] = v.w;
                sf[k] = c_ * c_;
            } else {
                // the relative vector as hi + lo when the search kept the low parts; r and 1/r to
                // about 2^-46
                const float4 vl = w.nb_vlo ? w.nb_vlo[sb + k] : make_float4(0.f, 0.f, 0.f, 0.f);
                float px, ex, py, ey, pz, ez, s1, e1, s2, e2;
                two_prod(v.x, v.x, px, ex);
                two_prod(v.y, v.y, py, ey);
                two_prod(v.z, v.z, pz, ez);
                ex = fmaf(2.f * v.x, vl.x, ex);
                ey = fmaf(2.f * v.y, vl.y, ey);
                ez = fmaf(2.f * v.z, vl.z, ez);
                two_sum(px, py, s1, e1);
                two_sum(s1, pz, s2, e2);
                const float r2l = ((e1 + e2) + (ex + ey)) + ez;
                const float rh = sqrtf(s2);
                const float rl = (fmaf(-rh, rh, s2) + r2l) * (0.5f / rh);
                const float ih = 1.f / rh;
                const float il = ih * (fmaf(-rh, ih, 1.f) - rl * ih);
                const float hx = __fmul_rn(v.x, ih), hy = __fmul_rn(v.y, ih), hz = __fmul_rn(v.z, ih);
                sv[k] = make_float4(hx, hy, hz, rh);
                const float c_ = cospif(0.5f * (rh / d.rc));
                sl[k] = make_float4(fmaf(v.x, ih, -hx) + fmaf(v.x, il, vl.x * ih),
                                    fmaf(v.y, ih, -hy) + fmaf(v.y, il, vl.y * ih),
                                    fmaf(v.z, ih, -hz) + fmaf(v.z, il, vl.z * ih), c_ * c_);
            }
        }
        species_segments(d, w.nb_idx + sb, n, seg, lane);
        sync();

        if (TEAM) {
            // radial terms: eight lanes per species and shell, each every eighth entry
            const int items = d.S * d.n_rad;
            for (int x0 = rank * (threads / 8); x0 < items; x0 += ctas * (threads / 8)) {
                const int x = x0 + tid / 8, sp = x / d.n_rad, nn = x - sp * d.n_rad;
                float acc = 0.f;
                if (x < items) {
                    const float rs = d.rs_rad[nn];
                    for (int k = seg[sp] + (tid & 7); k < seg[sp + 1]; k += 8) {
                        const float xr = sv[k].w - rs;
                        acc = fmaf(ex2f(-eta_rl * (xr * xr)), sl[k].w, acc);
                    }
                }
#pragma unroll
                for (int o = 4; o >= 1; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
                if (x < items && (tid & 7) == 0) put((size_t)row * d.D + x, acc);
            }
        }
        // radial terms: lanes over shells
        for (int nn = lane; !TEAM && nn < d.n_rad; nn += 32) {
            const float rs = d.rs_rad[nn];
            for (int sp = 0; sp < d.S; ++sp) {
                float acc = 0.f;
                for (int k = seg[sp]; k < seg[sp + 1]; ++k) {
                    const float xr = (FAST ? sr[k] : sv[k].w) - rs;
                    acc = fmaf(ex2f(-eta_rl * (xr * xr)), FAST ? sf[k] : sl[k].w, acc);
                }
                put((size_t)row * d.D + sp * d.n_rad + nn, acc);
            }
        }

        // angular terms: CM sector chunks of 8 and one shell chunk of 8 at a time
        for (int u0 = 0; u0 < ncm * ncn; u0 += CM) {
            const int m0 = (u0 % ncm) * 8, n0 = (u0 / ncm) * 8;   // CM divides ncm
            float2 chm[CM], shm[CM], tan_m[FAST ? 1 : CM];
#pragma unroll
            for (int mc = 0; mc < CM; ++mc) {
                const int m = min(m0 + mc * 8 + g, d.n_theta - 1);
                chm[mc] = dup(d.chr_t[m]);
                shm[mc] = dup(d.shr_t[m]);
                if (!FAST) tan_m[mc] = dup(d.tan_t[m]);
            }
            const float rs_g = d.rs_ang[min(n0 + g, d.n_ang_r - 1)];
            const float2 nR = dup(FAST ? (r_c - rs_g) * s_eta : -rs_g);
            const float2 y0 = dup(1.f + d.r_half), nk0 = dup(-d.r_half);
            // the factor 2 of A_m = 2 y_m^zeta; FAST: and what rounding 1 + (R - 1)/2 takes from y^zeta
            // where it is not small (y near 1)
            const float two = FAST ? fmaf(2.f * d.zeta, d.r_half - (y0.x - 1.f), 2.f) : 2.f;
            const float2 me = dup(-d.eta_ang * 1.4426950408889634f);
            // rows g (A_hi) and g + 8 (A_lo), shells 2 t and 2 t + 1 of a block's sums
            auto flush = [&](int blk, const float (&acc)[CM][4]) {
#pragma unroll
                for (int mc = 0; mc < CM; ++mc) {
                    const int m = m0 + mc * 8 + g, nq = n0 + 2 * t;
                    const float v0 = two * (acc[mc][0] + acc[mc][2]), v1 = two * (acc[mc][1] + acc[mc][3]);
                    const size_t o = (size_t)row * d.D + d.rad_cols + blk * nbins + m * d.n_ang_r + nq;
                    if (m < d.n_theta) {
                        if (even && nq < d.n_ang_r) {
                            put2(o, v0, v1);
                        } else {
                            if (nq < d.n_ang_r) put(o, v0);
                            if (nq + 1 < d.n_ang_r) put(o + 1, v1);
                        }
                    }
                }
            };
            auto put_part = [&](const float (&v)[CM][4], float4* to) {
#pragma unroll
                for (int mc = 0; mc < CM; ++mc) to[mc * 32 + lane] = make_float4(v[mc][0], v[mc][1], v[mc][2], v[mc][3]);
            };
            auto add_part = [&](float (&v)[CM][4], const float4* from) {
#pragma unroll
                for (int mc = 0; mc < CM; ++mc) {
                    const float4 x = from[mc * 32 + lane];
                    v[mc][0] += x.x; v[mc][1] += x.y; v[mc][2] += x.z; v[mc][3] += x.w;
                }
            };
            TeamRounds rounds(d, seg, wt, team);   // not TEAM: unused
            // TEAM: block that later warps share, the end of its rounds; that of a block begun by earlier ones
            int open = -1, open_end = 0, cont_end = 0;
            int blk = 0;
            float acc[CM][4], comp[FAST ? 1 : CM][4];
            for (int a = 0; a < d.S; ++a)
                for (int b = a; b < d.S; ++b, ++blk) {
                    int first = 0, last = 0;
                    if (TEAM) {
                        const int np = TeamRounds::block_pairs(seg, a, b);
                        rounds.next(np, first, last);
                        if (np == 0 && wt == 0) {
                            const float zero[CM][4] = {};
                            flush(blk, zero);
                        }
                        if (first >= last) continue;
                    }
                    BlockPairs bp(seg[a], seg[a + 1] - seg[a], seg[b], seg[b + 1] - seg[b], a == b,
                                  lane + 32 * first);
                    const int end = TEAM ? min(bp.n, 32 * last) : bp.n;
#pragma unroll
                    for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[mc][q] = comp[FAST ? 0 : mc][q] = 0.f;
                    for (int p0 = 32 * first; p0 < end; p0 += 32, bp.next()) {
                        // step 1: geometry of the lane's pair (weight 0 past the block's end)
                        {
                            const bool on = p0 + lane < bp.n;
                            int k1, k2;
                            bp.get(on, k1, k2);
                            const float4 va = sv[k1], vb = sv[k2];
                            if (FAST) {
                                const float wx = fmaf(va.y, vb.z, -va.z * vb.y);
                                const float wy = fmaf(va.z, vb.x, -va.x * vb.z);
                                const float wz = fmaf(va.x, vb.y, -va.y * vb.x);
                                const float c = fmaf(va.x, vb.x, fmaf(va.y, vb.y, va.z * vb.z));
                                const float s2 = fmaf(wx, wx, fmaf(wy, wy, fmaf(wz, wz, d.eps_theta)));
                                float sh, ch;
                                half_angles<true>(d, c, s2, sh, ch);
                                pa_f[off0] = sh;
                                pa_f[off1] = ch;
                                pr_f[off0] = va.w + vb.w;
                                pr_f[off1] = on ? sf[k1] * sf[k2] : 0.f;
                            } else {
                                const float4 la = sl[k1], lb = sl[k2];
                                // cos = u1 . u2 as hi + lo
                                float p0_, e0, p1_, e1, p2_, e2, s, ea, c, eb;
                                two_prod(va.x, vb.x, p0_, e0);
                                two_prod(va.y, vb.y, p1_, e1);
                                two_prod(va.z, vb.z, p2_, e2);
                                two_sum(p0_, p1_, s, ea);
                                two_sum(s, p2_, c, eb);
                                const float cross = fmaf(va.x, lb.x, fmaf(la.x, vb.x, fmaf(va.y, lb.y,
                                                    fmaf(la.y, vb.y, fmaf(va.z, lb.z, la.z * vb.z)))));
                                // cos th' = cos / R
                                const float cl = fmaf(-c, d.r_def, (((ea + eb) + (e0 + e1)) + e2) + cross);
                                // sin, cos of th'/2 as hi + lo: square roots of (1 -/+ cos th')/2
                                float sh, shl, ch, chl;
                                half_pair(-c, -cl, sh, shl);
                                half_pair(c, cl, ch, chl);
                                float rbh, rbl;
                                rbar_halves(va.w, vb.w, rbh, rbl);
                                pa_f[off0] = sh;
                                pa_f[off1] = ch;
                                pr_f[off0] = rbh;
                                pr_f[off1] = rbl;
                                pd_f[off0] = fmaf(shl, ch, -chl * sh);
                                pd_f[off1] = on ? la.w * lb.w : 0.f;
                            }
                        }
                        __syncwarp();
                        // step 2: groups of 8 pairs
                        float c[CM][4];
#pragma unroll
                        for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                            for (int q = 0; q < 4; ++q) c[mc][q] = 0.f;
                        float q2[FAST ? 1 : CM][4];
                        const int left = bp.n - p0;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (8 * k >= left) break;
                            float4 ha = pa[4 * k + t], hr = pr[4 * k + t], hd;
                            if (!FAST) hd = pd[4 * k + t];
                            if (k >= 2) {
                                ha = make_float4(ha.z, ha.w, ha.x, ha.y);
                                hr = make_float4(hr.z, hr.w, hr.x, hr.y);
                                if (!FAST) hd = make_float4(hd.z, hd.w, hd.x, hd.y);
                            }
                            const float2 sh = make_float2(ha.x, ha.y), ch = make_float2(ha.z, ha.w);
                            float2 z, ff;
                            if (FAST) {
                                const float2 x = __fadd2_rn(make_float2(hr.x, hr.y), nR);
                                z = __fmul2_rn(x, make_float2(-x.x, -x.y));
                                ff = make_float2(hr.z, hr.w);
                            } else {
                                const float2 x = __fadd2_rn(__fadd2_rn(make_float2(hr.x, hr.y), nR),
                                                            make_float2(hr.z, hr.w));
                                z = __fmul2_rn(__fmul2_rn(x, x), me);
                                ff = make_float2(hd.z, hd.w);
                            }
                            const float2 e = __fmul2_rn(make_float2(ex2f(z.x), ex2f(z.y)), ff);
                            float2 eh, el;
                            tf_split<!FAST>(e, eh, el);
#pragma unroll
                            for (int mc = 0; mc < CM; ++mc) {
                                const float2 w2 = __fmul2_rn(ch, shm[mc]);
                                float2 ee = __ffma2_rn(sh, chm[mc], make_float2(-w2.x, -w2.y));
                                if (FAST) {
                                    const float2 A = pow2_y(d.zeta, __ffma2_rn(ee, make_float2(-ee.x, -ee.y), y0));
                                    // scalar differences: the operand quad interleaves hi and lo
                                    const float a0 = tf_hi(A.x), a1 = tf_hi(A.y), l0 = A.x - a0, l1 = A.y - a1;
                                    mma8(c[mc], a0, l0, a1, l1, eh.x, eh.y);
                                    mma8(c[mc], a0, l0, a1, l1, el.x, el.y);
                                } else {
                                    const float2 mch = make_float2(-ch.x, -ch.y);
                                    const float2 dw = __ffma2_rn(mch, shm[mc], w2);   // minus the rounding of w2
                                    const float2 cc = __ffma2_rn(ch, chm[mc], __fmul2_rn(sh, shm[mc]));
                                    const float2 dt = __fadd2_rn(make_float2(hd.x, hd.y), tan_m[mc]);
                                    ee = __fadd2_rn(ee, __ffma2_rn(dt, cc, dw));
                                    const float2 A = pow2_t<PW, true>(d.zlog, d.zeta, __ffma2_rn(ee, ee, nk0));
                                    float2 Ah, Al;
                                    tf_split<true>(A, Ah, Al);
                                    // the tensor cores truncate their sums: two groups deep here, one where
                                    // a small exponent makes the terms of a block alike in size, so that what
                                    // is lost does not average out (zeta <= 8: 1.03 to 1.06 times the blocked
                                    // kernel's error with two, 0.93 to 1.01 with one, the same time)
                                    constexpr int deep = PW ? 2 : 1;
                                    if (k % deep) mma8(q2[mc], Ah.x, Al.x, Ah.y, Al.y, el.x, el.y);
                                    else mma8z(q2[mc], Ah.x, Al.x, Ah.y, Al.y, el.x, el.y);
                                    mma8(q2[mc], Ah.x, Al.x, Ah.y, Al.y, eh.x, eh.y);
                                    if (k % deep == deep - 1 || 8 * (k + 1) >= left) {
#pragma unroll
                                        for (int j = 0; j < 4; ++j) c[mc][j] += q2[mc][j];
                                    }
                                }
                            }
                        }
#pragma unroll
                        for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                if (FAST) {
                                    acc[mc][q] += c[mc][q];
                                } else {   // compensated sum over the block's rounds
                                    const float v = c[mc][q] - comp[FAST ? 0 : mc][q], ns = acc[mc][q] + v;
                                    comp[FAST ? 0 : mc][q] = (ns - acc[mc][q]) - v;
                                    acc[mc][q] = ns;
                                }
                            }
                        __syncwarp();
                    }
                    if (TEAM && first > 0) {
                        put_part(acc, part);
                        cont_end = rounds.rb;
                    } else if (TEAM && 32 * last < bp.n) {
                        open = blk;   // the warp's last block: its sums stay in acc
                        open_end = rounds.rb;
                    } else {
                        flush(blk, acc);
                    }
                }
            if (TEAM) {
                // sums of the CTA's warps after this one in the block that ends before round `end`
                const int R = rounds.R;
                auto add_later = [&](int end) {
                    for (int j = wt + 1; j < (rank + 1) * warps && R * j / team < end; ++j) {
                        if (R * j / team == R * (j + 1) / team) continue;   // no rounds
                        add_part(acc, part + (j - wt) * (int)(w_bytes / 16));
                    }
                };
                __syncthreads();
                if (open >= 0) add_later(open_end);
                if (cont_end > 0 && R * (rank * warps) / team == rounds.lo) {
                    // begun by an earlier CTA: the CTA's sum where its warp 0 would leave its part
                    // (that of this warp, or of one without rounds)
                    float sum[CM][4] = {};
                    for (int j = wt; j < (rank + 1) * warps && R * j / team < cont_end; ++j)
                        if (R * j / team < R * (j + 1) / team) add_part(sum, part + (j - wt) * (int)(w_bytes / 16));
                    put_part(sum, part - warp * (int)(w_bytes / 16));
                }
                cluster_sync();
                if (open >= 0) {
                    for (int q = rank + 1; q < ctas && R * (q * warps) / team < open_end; ++q)
                        if (R * (q * warps) / team < R * ((q + 1) * warps) / team)
                            add_part(acc, cg::this_cluster().map_shared_rank(part - warp * (int)(w_bytes / 16), q));
                    flush(open, acc);
                }
                cluster_sync();   // the parts are free again
            }
        }
    }
}

// ------------------------------------------------------------------ tangent

// Change of the descriptors along displacements u of the atoms (FAST arithmetic; the tangent feeds the
// weight gradient only).  With dcos, dr1, dr2 the changes of a pair's angle and distances, its term
// T_mn = 2 y_m^zeta E_n F (F = f_c f_c) changes by
//   Q_m (a E_n) + U_m E_n (b + c x_n),   U = y^zeta, Q = y^(zeta - 1) sin_eps dy/dcos,
//   a = 2 zeta F dcos / sin_eps,  b = 2 dF,  c x = -4 eta F dr_bar (r_bar - R_n):
// two outer products over the pairs on the tensor cores, with the roles of k_desc_mma's lanes.  An entry is
// staged with the change of its unit vector, m = (du - u dr) / r, so that dcos = m1 . u2 + u1 . m2.
// Bound: instruction issue, as the descriptor.  Against the fastest lane-per-pair kernel: 1024 molecules
// (17,396 atoms) 139 -> 81 us, 850 atoms in 50 molecules 29 -> 15 us.
__host__ __device__ inline size_t jvp_mma_bytes(int cap)
{
    return (size_t)((cap + 3) & ~3) * (16 + 16 + 8 + 4) + 16 * (16 + 16 + 16);
}

template <int CM>
__global__ void __launch_bounds__(kMW * 32, CM == 1 ? 6 : 5)
k_jvp_mma(DescDev d, Work w, const float* __restrict__ u, float* __restrict__ out)
{
    extern __shared__ float4 sm4[];
    __shared__ int s_seg[kMW][kMaxSpecies + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cap = w.cap, cap4 = (cap + 3) & ~3;
    char* base = reinterpret_cast<char*>(sm4) + (size_t)warp * jvp_mma_bytes(cap);
    float4* sv = reinterpret_cast<float4*>(base);   // unit vector, rho (see k_desc_mma)
    float4* sm = sv + cap4;                         // its change, dr
    float2* sx = reinterpret_cast<float2*>(sm + cap4);   // f_c, f_c'
    float* sr = reinterpret_cast<float*>(sx + cap4);
    float4* pa = reinterpret_cast<float4*>(sr + cap4);   // pairs t, t + 4 of a group: cos, sin_eps
    float4* pr = pa + 16;                                // rho, a
    float4* pd = pr + 16;                                // b, c
    const int slot = (lane >> 3) * 4 + t, half = (lane >> 2) & 1;
    const int off0 = slot * 4 + half + ((lane >> 4) << 1), off1 = slot * 4 + half + (2 - ((lane >> 4) << 1));
    float* pa_f = reinterpret_cast<float*>(pa);
    float* pr_f = reinterpret_cast<float*>(pr);
    float* pd_f = reinterpret_cast<float*>(pd);
    int* seg = s_seg[warp];
    const int ncm = (d.n_theta + 7) / 8, ncn = (d.n_ang_r + 7) / 8;
    const int nbins = d.n_theta * d.n_ang_r;
    const float r_c = d.rs_ang[d.n_ang_r / 2], s_eta = sqrtf(d.eta_ang * 1.4426950408889634f);
    const float c_x = -1.3862943611f * s_eta, eta_rl = d.eta_rad * 1.4426950408889634f;
    const bool even = ((d.D | d.rad_cols | d.n_ang_r) & 1) == 0;
    for (int64_t i = (int64_t)blockIdx.x * kMW + warp; i < w.N; i += (int64_t)gridDim.x * kMW) {
        const int64_t row = w.row_of_atom[i];
        if (row < 0) continue;   // ghosts are not centres
        const int n = w.nb_count[i];
        const size_t sb = (size_t)i * cap;
        const float ux = u[3 * i], uy = u[3 * i + 1], uz = u[3 * i + 2];
        __syncwarp();   // the previous atom's reads of the staging area are done
        for (int k = lane; k < n; k += 32) {
            const float4 v = w.nb_vec[sb + k];
            const int64_t j = w.nb_idx[sb + k].x;
            const float ir = 1.f / v.w;
            const float a = v.x * ir, b = v.y * ir, c = v.z * ir;
            const float dx = u[3 * j] - ux, dy = u[3 * j + 1] - uy, dz = u[3 * j + 2] - uz;
            const float dr = fmaf(a, dx, fmaf(b, dy, c * dz));
            float s_, c_;
            sincospif(0.5f * (v.w / d.rc), &s_, &c_);
            sv[k] = make_float4(a, b, c, (v.w - r_c) * (0.5f * s_eta));
            sm[k] = make_float4(fmaf(-a, dr, dx) * ir, fmaf(-b, dr, dy) * ir, fmaf(-c, dr, dz) * ir, dr);
            sx[k] = make_float2(c_ * c_, -d.pi_rc * s_ * c_);
            sr[k] = v.w;
        }
        species_segments(d, w.nb_idx + sb, n, seg, lane);
        __syncwarp();

        // radial terms: lanes over shells
        for (int nn = lane; nn < d.n_rad; nn += 32) {
            const float rs = d.rs_rad[nn];
            for (int sp = 0; sp < d.S; ++sp) {
                float acc = 0.f;
                for (int k = seg[sp]; k < seg[sp + 1]; ++k) {
                    const float xr = sr[k] - rs;
                    const float2 f = sx[k];
                    acc = fmaf(ex2f(-eta_rl * (xr * xr)) * sm[k].w, fmaf(-2.f * d.eta_rad * xr, f.x, f.y), acc);
                }
                out[(size_t)row * d.D + sp * d.n_rad + nn] = acc;
            }
        }

        // angular terms: CM sector chunks of 8 and one shell chunk of 8 at a time
        for (int u0 = 0; u0 < ncm * ncn; u0 += CM) {
            const int m0 = (u0 % ncm) * 8, n0 = (u0 / ncm) * 8;   // CM divides ncm
            float2 chm[CM], shm[CM];
#pragma unroll
            for (int mc = 0; mc < CM; ++mc) {
                const int m = min(m0 + mc * 8 + g, d.n_theta - 1);
                chm[mc] = dup(d.half_cos_t[m]);
                shm[mc] = dup(d.half_sin_t[m]);
            }
            const float2 nR = dup((r_c - d.rs_ang[min(n0 + g, d.n_ang_r - 1)]) * s_eta);
            int blk = 0;
            for (int a = 0; a < d.S; ++a)
                for (int b = a; b < d.S; ++b, ++blk) {
                    BlockPairs bp(seg[a], seg[a + 1] - seg[a], seg[b], seg[b + 1] - seg[b], a == b, lane);
                    float acc[CM][4];
#pragma unroll
                    for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                        for (int q = 0; q < 4; ++q) acc[mc][q] = 0.f;
                    for (int p0 = 0; p0 < bp.n; p0 += 32, bp.next()) {
                        // step 1: geometry of the lane's pair (weights 0 past the block's end)
                        {
                            const bool on = p0 + lane < bp.n;
                            int k1, k2;
                            bp.get(on, k1, k2);
                            const float4 va = sv[k1], vb = sv[k2], ma = sm[k1], mb = sm[k2];
                            const float2 f1 = sx[k1], f2 = sx[k2];
                            const float wx = fmaf(va.y, vb.z, -va.z * vb.y);
                            const float wy = fmaf(va.z, vb.x, -va.x * vb.z);
                            const float wz = fmaf(va.x, vb.y, -va.y * vb.x);
                            const float s2 = fmaf(wx, wx, fmaf(wy, wy, fmaf(wz, wz, d.eps_theta)));
                            const float ise = rsqf(fmaxf(s2, 1e-37f));
                            const float dc = fmaf(ma.x, vb.x, fmaf(ma.y, vb.y, ma.z * vb.z)) +
                                             fmaf(va.x, mb.x, fmaf(va.y, mb.y, va.z * mb.z));
                            const float F = on ? f1.x * f2.x : 0.f;
                            const float dF = on ? fmaf(f1.y * ma.w, f2.x, f1.x * f2.y * mb.w) : 0.f;
                            pa_f[off0] = fmaf(va.x, vb.x, fmaf(va.y, vb.y, va.z * vb.z));
                            pa_f[off1] = s2 * ise;
                            pr_f[off0] = va.w + vb.w;
                            pr_f[off1] = 2.f * d.zeta * F * ise * dc;
                            pd_f[off0] = 2.f * dF;
                            pd_f[off1] = c_x * F * (ma.w + mb.w);
                        }
                        __syncwarp();
                        // step 2: groups of 8 pairs
                        const int left = bp.n - p0;
                        float c[CM][4];
#pragma unroll
                        for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                            for (int q = 0; q < 4; ++q) c[mc][q] = 0.f;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            if (8 * k >= left) break;
                            float4 ha = pa[4 * k + t], hr = pr[4 * k + t], hd = pd[4 * k + t];
                            if (k >= 2) {
                                ha = make_float4(ha.z, ha.w, ha.x, ha.y);
                                hr = make_float4(hr.z, hr.w, hr.x, hr.y);
                                hd = make_float4(hd.z, hd.w, hd.x, hd.y);
                            }
                            const float2 cs = make_float2(ha.x, ha.y), se = make_float2(ha.z, ha.w);
                            const float2 x = __fadd2_rn(make_float2(hr.x, hr.y), nR);
                            const float2 z = __fmul2_rn(x, make_float2(-x.x, -x.y));
                            const float2 e = make_float2(ex2f(z.x), ex2f(z.y));
                            float2 qh, ql, rh, rl;
                            tf_split<false>(__fmul2_rn(e, make_float2(hr.z, hr.w)), qh, ql);
                            tf_split<false>(__fmul2_rn(e, __ffma2_rn(make_float2(hd.z, hd.w), x, make_float2(hd.x, hd.y))),
                                            rh, rl);
#pragma unroll
                            for (int mc = 0; mc < CM; ++mc) {
                                const float2 y = __ffma2_rn(cs, chm[mc], __ffma2_rn(se, shm[mc], dup(0.5f)));
                                const float2 ef = __ffma2_rn(se, chm[mc], __fmul2_rn(make_float2(-cs.x, -cs.y), shm[mc]));
                                const float2 p1 = pow2_y(d.zeta - 1.f, y);
                                const float2 U = __fmul2_rn(p1, y), Q = __fmul2_rn(p1, ef);
                                const float q0 = tf_hi(Q.x), q1 = tf_hi(Q.y), v0 = tf_hi(U.x), v1 = tf_hi(U.y);
                                mma8(c[mc], q0, Q.x - q0, q1, Q.y - q1, ql.x, ql.y);
                                mma8(c[mc], v0, U.x - v0, v1, U.y - v1, rl.x, rl.y);
                                mma8(c[mc], q0, Q.x - q0, q1, Q.y - q1, qh.x, qh.y);
                                mma8(c[mc], v0, U.x - v0, v1, U.y - v1, rh.x, rh.y);
                            }
                        }
#pragma unroll
                        for (int mc = 0; mc < CM; ++mc)
#pragma unroll
                            for (int q = 0; q < 4; ++q) acc[mc][q] += c[mc][q];
                        __syncwarp();
                    }
                    // rows g (hi) and g + 8 (lo), shells 2 t and 2 t + 1
#pragma unroll
                    for (int mc = 0; mc < CM; ++mc) {
                        const int m = m0 + mc * 8 + g, nq = n0 + 2 * t;
                        const float v0 = acc[mc][0] + acc[mc][2], v1 = acc[mc][1] + acc[mc][3];
                        float* o = out + (size_t)row * d.D + d.rad_cols + blk * nbins + m * d.n_ang_r + nq;
                        if (m >= d.n_theta) continue;
                        if (even && nq < d.n_ang_r) {
                            *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
                        } else {
                            if (nq < d.n_ang_r) o[0] = v0;
                            if (nq + 1 < d.n_ang_r) o[1] = v1;
                        }
                    }
                }
        }
    }
}

// ------------------------------------------------------------------ adjoint

// Gradient of sum_i g_i . G_i with respect to the neighbour vectors, as k_adj_cd of descriptor.cu,
// with the products T e and T (x e) of a species block's gradient tile T (sectors x shells) on the
// tensor cores: 16 pairs are the rows of one A operand (their Gaussians, evaluated by lane (g, t) for
// pairs g, g + 8 and shells t, t + 4), T^T the B operand, held in registers for the whole block.
// The result leaves sectors 2t, 2t + 1 of pairs g, g + 8 in lane (g, t), which evaluates those
// sectors' powers and multiplies; the four lanes of a pair leave their sums in shared memory for
// the pair's own lane, which applies the chain rule (step 3).
//
// Per-entry sums.  dc/dv1 = (W x v1)/(r1^3 r2), dc/dv2 = -(W x v2)/(r1 r2^3) with W = v1 x v2, so one
// vector X = (dT/dc) W/(r1 r2) serves both entries of a pair: q_k = (sum X) x v_k / r_k^2 (minus for
// second entries) plus the distance terms along v_k.  Each pair adds one float4 (X, dT/dr) to each of
// its entries; the positions of one diagonal of the block touch distinct entries, and the few
// diagonals within a round of 32 pairs go to different copies of the sums (nc of them), so nothing
// needs atomics and every sum has a fixed order.

// Shared-memory traffic bounds the kernel next to instruction issue (a warp's load of 4 bytes per lane
// takes the SM's data path for a cycle, also when lanes share addresses), so the pair buffers carry
// single floats, f_c and f_c' stay in registers from step 1 to step 3, and FAST stages unit vectors.

//
// TEAM: as in the descriptor; each warp adds to copies of its own, which the CTAs and then the cluster's
// first CTA sum at the end.

struct AdjSmem {
    int sv, sx, sr, g, atom;            // byte offsets within an atom's area, its size
    int sq, pa, pr, pts, pt1, warp;     // and within a warp's
    int total(int warps) const { return atom + warps * warp; }
};
__host__ __device__ inline AdjSmem adj_mma_smem(const DescDev& d, int cap, int nc, bool fast)
{
    const int c2 = (cap + 1) & ~1, c4 = (cap + 3) & ~3;
    AdjSmem a;
    a.sv = 0;
    a.sx = a.sv + cap * 16;
    a.sr = a.sx + c2 * (fast ? 8 : 16);
    a.g = a.sr + (fast ? c4 * 4 : 0);
    a.atom = a.g + ((d.D + 3) & ~3) * 4;
    a.sq = 0;
    a.pa = a.sq + nc * cap * 16;
    a.pr = a.pa + 16 * 16;
    a.pts = a.pr + 16 * (fast ? 8 : 16);
    a.pt1 = a.pts + 128 * 8;
    a.warp = a.pt1 + 128 * 4;
    return a;
}

template <bool FAST, int CM, int PW, bool TEAM>
__global__ void __launch_bounds__((TEAM ? kTeamMax : kMW) * 32, TEAM ? 2 : CM == 1 ? 5 : 4)
k_adj_mma(DescDev d, Work w, const float* __restrict__ g_rows, float* __restrict__ F, float* __restrict__ vir_atom,
          int nc)
{
    extern __shared__ float4 sm4[];
    __shared__ int s_seg[TEAM ? kTeamMax : kMW][kMaxSpecies + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int cap = w.cap;
    const int warps = TEAM ? blockDim.x >> 5 : 1, tid = TEAM ? threadIdx.x : lane, threads = 32 * warps;
    const int ctas = TEAM ? cg::this_cluster().num_blocks() : 1, rank = TEAM ? cg::this_cluster().block_rank() : 0;
    const int wt = TEAM ? rank * warps + warp : 0, team = ctas * warps;   // its number among the atom's warps
    const AdjSmem lay = adj_mma_smem(d, cap, nc, FAST);
    char* base = reinterpret_cast<char*>(sm4) + (TEAM ? 0 : (size_t)warp * (lay.atom + lay.warp));
    char* base_w = base + lay.atom + (TEAM ? warp * lay.warp : 0);
    auto sync = [&] {
        if (!TEAM) __syncwarp();
        else if (ctas > 1) cg::this_cluster().sync();
        else __syncthreads();
    };
    float4* sv = reinterpret_cast<float4*>(base + lay.sv);   // FAST: (unit vector, rho), else (v, r)
    float2* sx2 = reinterpret_cast<float2*>(base + lay.sx);  // FAST: (f_c, f_c')
    float4* sx4 = reinterpret_cast<float4*>(base + lay.sx);  // else (f_c, f_c', 1/r, -)
    float* sr = reinterpret_cast<float*>(base + lay.sr);     // FAST: r
    float4* sq = reinterpret_cast<float4*>(base_w + lay.sq); // nc copies of (sum X, sum dT/dr)
    float* sg = reinterpret_cast<float*>(base + lay.g);      // the atom's gradient row
    float4* pa = reinterpret_cast<float4*>(base_w + lay.pa); // pairs p, p + 8: sin, cos of th'/2 (FAST: cos, sin_eps)
    float2* pr2 = reinterpret_cast<float2*>(base_w + lay.pr);  // pairs p, p + 8: FAST distance,
    float4* pr4 = reinterpret_cast<float4*>(base_w + lay.pr);  // else its hi and lo parts
    float2* pts = reinterpret_cast<float2*>(base_w + lay.pts); // the four lanes' parts of a pair's sums
    float* pt1 = reinterpret_cast<float*>(base_w + lay.pt1);
    const int my = (lane >> 4) * 8 + (lane & 7), half = (lane >> 3) & 1;
    float* pa_my = reinterpret_cast<float*>(pa) + my * 4 + half;
    float* pr_my = reinterpret_cast<float*>(pr2) + my * (FAST ? 2 : 4) + half;
    int* seg = s_seg[warp];
    const int nbins = d.n_theta * d.n_ang_r;
    const float eta_l = d.eta_ang * 1.4426950408889634f;
    const float r_c = d.rs_ang[d.n_ang_r / 2], s_eta = sqrtf(eta_l);
    // this lane's shells (t, t + 4) and sectors (2t, 2t + 1 of each chunk)
    float2 nR0, nR1, chm[CM], shm[CM];
    {
        const float ra = d.rs_ang[min(t, d.n_ang_r - 1)], rb = d.rs_ang[min(t + 4, d.n_ang_r - 1)];
        nR0 = dup(FAST ? (r_c - ra) * s_eta : -ra);
        nR1 = dup(FAST ? (r_c - rb) * s_eta : -rb);
#pragma unroll
        for (int mc = 0; mc < CM; ++mc) {
            const int ma = min(mc * 8 + 2 * t, d.n_theta - 1), mb = min(mc * 8 + 2 * t + 1, d.n_theta - 1);
            chm[mc] = FAST ? make_float2(d.half_cos_t[ma], d.half_cos_t[mb]) : make_float2(d.chr_t[ma], d.chr_t[mb]);
            shm[mc] = FAST ? make_float2(d.half_sin_t[ma], d.half_sin_t[mb]) : make_float2(d.shr_t[ma], d.shr_t[mb]);
        }
    }
    // dT/dr = s1 Fp S1 + ...: x e in the units of nR0
    const float s1 = FAST ? -1.3862943611f * s_eta : -2.f * d.eta_ang;   // -2 eta / s_eta, s_eta^2 = eta log2(e)
    const bool gvec = (d.D & 3) == 0 && (reinterpret_cast<uintptr_t>(g_rows) & 15) == 0;

    for (int64_t i = TEAM ? blockIdx.x / ctas : (int64_t)blockIdx.x * kMW + warp; i < w.N;
         i += TEAM ? gridDim.x / ctas : (int64_t)gridDim.x * kMW) {
        const int64_t row = w.row_of_atom[i];
        if (row < 0) continue;   // ghosts are not centres
        const int n = w.nb_count[i];
        const size_t sb = (size_t)i * cap;
        sync();   // the previous atom's reads of the staging area are done
        {
            const float* gi = g_rows + (size_t)row * d.D;
            if (gvec) {
                for (int c = tid; c < d.D / 4; c += threads)
                    reinterpret_cast<float4*>(sg)[c] = reinterpret_cast<const float4*>(gi)[c];
            } else {
                for (int c = tid; c < d.D; c += threads) sg[c] = gi[c];
            }
        }
        for (int k = tid; k < n; k += threads) {
            const float4 v = w.nb_vec[sb + k];
            const float ir = 1.f / v.w;
            float s_, c_;
            sincospif(0.5f * (v.w / d.rc), &s_, &c_);
            const float fc = c_ * c_, dfc = -d.pi_rc * s_ * c_;
            if (FAST) {
                sv[k] = make_float4(v.x * ir, v.y * ir, v.z * ir, (v.w - r_c) * (0.5f * s_eta));
                sx2[k] = make_float2(fc, dfc);
                sr[k] = v.w;
            } else {
                sv[k] = v;
                sx4[k] = make_float4(fc, dfc, ir, 0.f);
            }
        }
        for (int c = 0; c < nc; ++c)
            for (int k = lane; k < n; k += 32) sq[c * cap + k] = make_float4(0.f, 0.f, 0.f, 0.f);
        species_segments(d, w.nb_idx + sb, n, seg, lane);
        if (TEAM) __syncthreads();
        else __syncwarp();

        // radial terms: four lanes per entry, each every fourth shell
        for (int k0 = 8 * wt; k0 < n; k0 += 8 * team) {
            const int k = k0 + g;
            float T0 = 0.f, T1 = 0.f;
            if (k < n) {
                int sp = 0;
                while (k >= seg[sp + 1]) ++sp;
                const float* gr = sg + sp * d.n_rad;
                const float r = FAST ? sr[k] : sv[k].w, me = -d.eta_rad * 1.4426950408889634f;
                for (int nn = t; nn < d.n_rad; nn += 4) {
                    const float xr = r - d.rs_rad[nn];
                    const float ge = gr[nn] * ex2f(me * (xr * xr));
                    T0 += ge;
                    T1 = fmaf(ge, xr, T1);
                }
            }
            T0 += __shfl_xor_sync(0xffffffffu, T0, 1);
            T1 += __shfl_xor_sync(0xffffffffu, T1, 1);
            T0 += __shfl_xor_sync(0xffffffffu, T0, 2);
            T1 += __shfl_xor_sync(0xffffffffu, T1, 2);
            if (k < n && t == 0) {
                const float fc = FAST ? sx2[k].x : sx4[k].x, dfc = FAST ? sx2[k].y : sx4[k].y;
                sq[k].w = fmaf(dfc, T0, -2.f * d.eta_rad * fc * T1);   // the warp's own copy
            }
        }
        __syncwarp();

        TeamRounds rounds(d, seg, wt, team);   // not TEAM: unused
        int blk = 0;
        for (int a = 0; a < d.S; ++a)
            for (int b = a; b < d.S; ++b, ++blk) {
                int first = 0, last = 0;
                if (TEAM) {
                    rounds.next(TeamRounds::block_pairs(seg, a, b), first, last);
                    if (first >= last) continue;
                }
                BlockPairs bp(seg[a], seg[a + 1] - seg[a], seg[b], seg[b + 1] - seg[b], a == b, lane + 32 * first);
                const int end = TEAM ? min(bp.n, 32 * last) : bp.n;
                if (bp.n == 0) continue;
                // T^T as B operands (sector g, shells t and t + 4), hi and lo
                // FAST: and of T^T with its columns scaled by R - R_c (in the units of x)
                float2 th[CM], tl[CM], uh[FAST ? CM : 1], ul[FAST ? CM : 1];
#pragma unroll
                for (int mc = 0; mc < CM; ++mc) {
                    const int m = mc * 8 + g;
                    const float* gt = sg + d.rad_cols + blk * nbins + m * d.n_ang_r;
                    const bool in = m < d.n_theta;
                    const float2 T = make_float2(in && t < d.n_ang_r ? gt[t] : 0.f,
                                                 in && t + 4 < d.n_ang_r ? gt[t + 4] : 0.f);
                    tf_split<true>(T, th[mc], tl[mc]);
                    if (FAST) tf_split<true>(__fmul2_rn(T, make_float2(nR0.x, nR1.x)), uh[mc], ul[mc]);
                }
                for (int p0 = 32 * first; p0 < end; p0 += 32, bp.next()) {
                    // step 1: geometry of the lane's pair
                    const bool on = p0 + lane < bp.n;
                    int k1, k2;
                    bp.get(on, k1, k2);
                    float wx, wy, wz, ise;   // W/(r1 r2), 1/sin_eps
                    float2 f1, f2;           // (f_c, f_c') of the two entries
                    float rho = 0.f;
                    {
                        const float4 va = sv[k1], vb = sv[k2];
                        float sh, ch;
                        if (FAST) {
                            f1 = sx2[k1]; f2 = sx2[k2];
                            wx = fmaf(va.y, vb.z, -va.z * vb.y);
                            wy = fmaf(va.z, vb.x, -va.x * vb.z);
                            wz = fmaf(va.x, vb.y, -va.y * vb.x);
                            const float s2 = fmaf(wx, wx, fmaf(wy, wy, fmaf(wz, wz, d.eps_theta)));
                            ise = rsqf(fmaxf(s2, 1e-37f));
                            sh = fmaf(va.x, vb.x, fmaf(va.y, vb.y, va.z * vb.z));   // cos, sin_eps themselves
                            ch = s2 * ise;
                            rho = va.w + vb.w;
                            pr_my[0] = rho;
                        } else {
                            const float4 xa = sx4[k1], xb = sx4[k2];
                            f1 = make_float2(xa.x, xa.y);
                            f2 = make_float2(xb.x, xb.y);
                            const float ir12 = xa.z * xb.z;
                            wx = dop(va.y, vb.z, va.z, vb.y) * ir12;
                            wy = dop(va.z, vb.x, va.x, vb.z) * ir12;
                            wz = dop(va.x, vb.y, va.y, vb.x) * ir12;
                            const float s2 = fmaf(wx, wx, fmaf(wy, wy, fmaf(wz, wz, d.eps_theta)));
                            const float c = fmaf(va.x, vb.x, fmaf(va.y, vb.y, va.z * vb.z)) * ir12;
                            half_angles<false>(d, fminf(fmaxf(c, -1.f), 1.f), s2, sh, ch);
                            const float se = sqrt_nr(s2);
                            ise = se > 0.f ? div_nr(1.f, se) : 0.f;
                            float rbh, rbl;
                            rbar_halves(va.w, vb.w, rbh, rbl);
                            pr_my[0] = rbh;
                            pr_my[2] = rbl;
                        }
                        pa_my[0] = sh;
                        pa_my[2] = ch;
                    }
                    __syncwarp();
                    // step 2: groups of 16 pairs
                    const int left = bp.n - p0;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (16 * h >= left) break;
                        float2 x0, x1, z0, z1;
                        if (FAST) {
                            const float2 hr = pr2[8 * h + g];
                            x0 = __fadd2_rn(hr, nR0);
                            x1 = __fadd2_rn(hr, nR1);
                            z0 = __fmul2_rn(x0, make_float2(-x0.x, -x0.y));
                            z1 = __fmul2_rn(x1, make_float2(-x1.x, -x1.y));
                        } else {
                            const float4 hr = pr4[8 * h + g];
                            const float2 hi = make_float2(hr.x, hr.y), lo = make_float2(hr.z, hr.w);
                            x0 = __fadd2_rn(__fadd2_rn(hi, nR0), lo);
                            x1 = __fadd2_rn(__fadd2_rn(hi, nR1), lo);
                            z0 = __fmul2_rn(__fmul2_rn(x0, x0), dup(-eta_l));
                            z1 = __fmul2_rn(__fmul2_rn(x1, x1), dup(-eta_l));
                        }
                        const float2 e0 = make_float2(ex2f(z0.x), ex2f(z0.y)), e1 = make_float2(ex2f(z1.x), ex2f(z1.y));
                        float2 e0h, e0l, e1h, e1l, f0h, f0l, f1h, f1l;
                        tf_split<!FAST>(e0, e0h, e0l);
                        tf_split<!FAST>(e1, e1h, e1l);
                        if (!FAST) {
                            tf_split<true>(__fmul2_rn(x0, e0), f0h, f0l);
                            tf_split<true>(__fmul2_rn(x1, e1), f1h, f1l);
                        }
                        const float4 sc = pa[8 * h + g];   // sin of the two pairs, cos of the two pairs
                        float2 Tc[2], S0[2], S1[2];
#pragma unroll
                        for (int mc = 0; mc < CM; ++mc) {
                            float C[4], X[4];
                            mma8z(C, e0h.x, e0h.y, e1h.x, e1h.y, tl[mc].x, tl[mc].y);
                            mma8(C, e0l.x, e0l.y, e1l.x, e1l.y, th[mc].x, th[mc].y);
                            mma8(C, e0h.x, e0h.y, e1h.x, e1h.y, th[mc].x, th[mc].y);
                            if (FAST) {
                                // sum x T e = rho sum T e + sum (R_c - R) T e: rho enters in step 3
                                mma8z(X, e0h.x, e0h.y, e1h.x, e1h.y, ul[mc].x, ul[mc].y);
                                mma8(X, e0l.x, e0l.y, e1l.x, e1l.y, uh[mc].x, uh[mc].y);
                                mma8(X, e0h.x, e0h.y, e1h.x, e1h.y, uh[mc].x, uh[mc].y);
                            } else {
                                mma8z(X, f0h.x, f0h.y, f1h.x, f1h.y, tl[mc].x, tl[mc].y);
                                mma8(X, f0l.x, f0l.y, f1l.x, f1l.y, th[mc].x, th[mc].y);
                                mma8(X, f0h.x, f0h.y, f1h.x, f1h.y, th[mc].x, th[mc].y);
                            }
#pragma unroll
                            for (int P = 0; P < 2; ++P) {
                                const float2 sh2 = dup(P ? sc.y : sc.x), ch2 = dup(P ? sc.w : sc.z);
                                float2 y, p1, ef;   // y_m, y_m^(zeta - 1), sin_eps dy_m/dcos
                                if (FAST) {
                                    y = __ffma2_rn(sh2, chm[mc], __ffma2_rn(ch2, shm[mc], dup(0.5f)));
                                    ef = __ffma2_rn(ch2, chm[mc], __fmul2_rn(make_float2(-sh2.x, -sh2.y), shm[mc]));
                                    p1 = pow2_y(d.zeta - 1.f, y);
                                } else {
                                    const float2 ee = __ffma2_rn(sh2, chm[mc],
                                                                 __fmul2_rn(make_float2(-ch2.x, -ch2.y), shm[mc]));
                                    const float2 tt = __ffma2_rn(ee, ee, dup(-d.r_half));
                                    y = __fadd2_rn(dup(1.f), make_float2(-tt.x, -tt.y));
                                    ef = __fmul2_rn(ee, __ffma2_rn(ch2, chm[mc], __fmul2_rn(sh2, shm[mc])));
                                    p1 = pow2_t<PW, false>(d.zlog1, d.zeta - 1.f, tt);
                                }
                                const float2 U = __fmul2_rn(p1, y), Q = __fmul2_rn(p1, ef);
                                const float2 Cp = P ? make_float2(C[2], C[3]) : make_float2(C[0], C[1]);
                                const float2 Xp = P ? make_float2(X[2], X[3]) : make_float2(X[0], X[1]);
                                S0[P] = mc ? __ffma2_rn(U, Cp, S0[P]) : __fmul2_rn(U, Cp);
                                S1[P] = mc ? __ffma2_rn(U, Xp, S1[P]) : __fmul2_rn(U, Xp);
                                Tc[P] = mc ? __ffma2_rn(Q, Cp, Tc[P]) : __fmul2_rn(Q, Cp);
                            }
                        }
                        // slots permuted per part so that the lanes' stores fall on different banks
#pragma unroll
                        for (int P = 0; P < 2; ++P) {
                            const int p = 16 * h + 8 * P + g;
                            pts[t * 32 + (p ^ (4 * t))] = make_float2(Tc[P].x + Tc[P].y, S0[P].x + S0[P].y);
                            pt1[t * 32 + (p ^ (8 * t))] = S1[P].x + S1[P].y;
                        }
                    }
                    __syncwarp();
                    // step 3: chain rule of the lane's pair and its two entries' sums
                    float4 q1 = make_float4(0.f, 0.f, 0.f, 0.f);
                    float tr2 = 0.f;
                    if (on) {
                        float2 s = pts[lane];
                        float S1 = pt1[lane];
#pragma unroll
                        for (int j = 1; j < 4; ++j) {
                            s = __fadd2_rn(s, pts[j * 32 + (lane ^ (4 * j))]);
                            S1 += pt1[j * 32 + (lane ^ (8 * j))];
                        }
                        if (FAST) S1 = fmaf(rho, s.y, S1);
                        const float Fp = f1.x * f2.x;
                        const float dTc = 2.f * d.zeta * Fp * ise * s.x;   // dT/dcos
                        q1.x = dTc * wx;
                        q1.y = dTc * wy;
                        q1.z = dTc * wz;
                        const float sf = s1 * Fp * S1, S02 = 2.f * s.y;
                        q1.w = fmaf(f1.y * f2.x, S02, sf);                 // dT/dr1
                        tr2 = fmaf(f1.x * f2.y, S02, sf);                  // dT/dr2
                    }
                    const int q0 = __shfl_sync(0xffffffffu, bp.q, 0);
                    const int qd = bp.q - q0;                             // diagonal within the round
                    const int nd = __shfl_sync(0xffffffffu, bp.q, 31) - q0 + 1;
                    for (int c0 = 0; c0 < nd; c0 += nc) {
                        const bool act = on && qd >= c0 && qd < c0 + nc;
                        float4* cp = sq + (qd - c0) * cap;
                        if (act) {
                            float4 o = cp[k1];
                            cp[k1] = make_float4(o.x + q1.x, o.y + q1.y, o.z + q1.z, o.w + q1.w);
                        }
                        __syncwarp();
                        if (act) {
                            float4 o = cp[k2];
                            cp[k2] = make_float4(o.x - q1.x, o.y - q1.y, o.z - q1.z, o.w + tr2);
                        }
                        __syncwarp();
                    }
                }
            }

        // TEAM: the warps' copies into the CTA's first; warp 0 of the cluster's first CTA then has them all
        if (TEAM) {
            __syncthreads();
            for (int k = tid; k < n; k += threads) {
                float4* q0 = reinterpret_cast<float4*>(base + lay.atom + lay.sq) + k;
                float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int j = 0; j < warps; ++j) {
                    const float4* qj = reinterpret_cast<float4*>(base + lay.atom + j * lay.warp + lay.sq) + k;
                    for (int c = 0; c < nc; ++c) {
                        const float4 o = qj[c * cap];
                        z.x += o.x; z.y += o.y; z.z += o.z; z.w += o.w;
                    }
                }
                *q0 = z;
            }
            sync();
            if (wt > 0) continue;
        }

        // entries' gradients, scattered to the forces
        float fx = 0.f, fy = 0.f, fz = 0.f;
        float vv[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) vv[k] = 0.f;
        for (int k = lane; k < n; k += 32) {
            float4 z = sq[k];
            for (int c = 1; c < (TEAM ? ctas : nc); ++c) {
                const float4 o = TEAM ? cg::this_cluster().map_shared_rank(sq, c)[k] : sq[c * cap + k];
                z.x += o.x; z.y += o.y; z.z += o.z; z.w += o.w;
            }
            float4 v = sv[k];
            float q0, q1, q2;
            if (FAST) {
                // v is the unit vector: q = (Z x u) / r + T u
                const float r = sr[k], ir = rcpf(r);
                q0 = fmaf(z.w, v.x, fmaf(z.y, v.z, -z.z * v.y) * ir);
                q1 = fmaf(z.w, v.y, fmaf(z.z, v.x, -z.x * v.z) * ir);
                q2 = fmaf(z.w, v.z, fmaf(z.x, v.y, -z.y * v.x) * ir);
                v = make_float4(v.x * r, v.y * r, v.z * r, r);
            } else {
                const float ir = sx4[k].z, ir2 = ir * ir, tr = z.w * ir;
                q0 = fmaf(tr, v.x, dop(z.y, v.z, z.z, v.y) * ir2);
                q1 = fmaf(tr, v.y, dop(z.z, v.x, z.x, v.z) * ir2);
                q2 = fmaf(tr, v.z, dop(z.x, v.y, z.y, v.x) * ir2);
            }
            fx += q0; fy += q1; fz += q2;
            const int64_t j = w.nb_idx[sb + k].x;
            atomicAdd(&F[3 * j + 0], -q0);
            atomicAdd(&F[3 * j + 1], -q1);
            atomicAdd(&F[3 * j + 2], -q2);
            const float rv[3] = {v.x, v.y, v.z}, qq[3] = {q0, q1, q2};
#pragma unroll
            for (int aa = 0; aa < 3; ++aa)
#pragma unroll
                for (int bb = 0; bb < 3; ++bb) vv[3 * aa + bb] -= qq[aa] * rv[bb];
        }
        add_centre(w, i, fx, fy, fz, vv, F, vir_atom, lane);
    }
    if (TEAM) sync();   // the other CTAs' shared memory is read until here
}

// resident CTAs walking the atoms: as many as fit on the GPU at once, no more than the atoms need
template <class Kern, class... Args>
cudaError_t launch_resident(Kern kern, int64_t N, size_t smem, cudaStream_t s, Args... args)
{
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMW * 32, smem);
    if (e != cudaSuccess) return e;
    const unsigned nb = (unsigned)std::min<int64_t>((N + kMW - 1) / kMW, (int64_t)sm_count() * std::max(per_sm, 1));
    kern<<<nb, kMW * 32, smem, s>>>(args...);
    return cudaGetLastError();
}

// a cluster per atom (TEAM)
struct Team {
    int ctas, warps;   // CTAs per cluster, warps per CTA
};
template <class Kern, class... Args>
cudaError_t launch_team(Kern kern, int64_t N, Team tm, size_t smem, cudaStream_t s, Args... args)
{
    cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)tm.ctas;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(N * tm.ctas));
    cfg.blockDim = dim3((unsigned)tm.warps * 32);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

constexpr size_t kMaxSmem = 200 * 1024;

}  // namespace

// |y|^e in place of max(y, 0)^e: y is at least -(R - 1)/2, so below 0 this is at most ((R - 1)/2)^e, which
// has to stay below the hardware log2's error of the powers near 1 (zeta = 2: up to eps = 1.9e-6, zeta = 4: 0.03)
static bool no_clamp(const DescDev& d, float e) { return powf(d.r_half, e) <= 4.77e-7f; }
// FAST needs exponents for which the splits' truncation (descriptor) and |y|^e in place of the clamp at
// y = 0 (descriptor e = zeta, adjoint and tangent zeta - 1) stay below the hardware log2's error
static bool desc_fast(const DescDev& d, bool fast) { return fast && d.zeta >= 16.f && no_clamp(d, d.zeta); }
static bool adj_fast(const DescDev& d, bool fast) { return fast && d.zeta >= 2.f && no_clamp(d, d.zeta - 1.f); }
bool mma_fast(const DescDev& d, bool adjoint) { return adjoint ? adj_fast(d, true) : desc_fast(d, true); }
// Terms of the logarithm's series for (1 - t)^e, 0 for pow_low.  For t > 0 see the file comment; t is at least
// -(R - 1)/2, where dropping the terms from t^(k+1) on moves the power by e |t|^(k+1)/(k+1) of itself: 8 terms
// serve zeta = 50 up to eps = 0.4, at eps = 3 they were off by 1e-2
static int log_terms(const DescDev& d, float e)
{
    auto holds = [&](int k) { return e * powf(d.r_half, (float)(k + 1)) / (float)(k + 1) <= 1e-8f; };
    return e >= 32.f && holds(8) ? 8 : e >= 16.f && holds(13) ? 13 : 0;
}

static size_t desc_smem(const Work& w, const DescDev& d, bool fast)
{
    return kMW * (desc_fast(d, fast) ? desc_mma_atom_bytes<true>(w.cap) + desc_mma_warp_bytes<true>(0)
                                     : desc_mma_atom_bytes<false>(w.cap) + desc_mma_warp_bytes<false>(0));
}

// Warps per atom below kSplitAtoms atoms, where one warp each leaves SMs idle and its chain of rounds is the
// kernel's time (descriptor / adjoint, us): 16 carbon atoms 117 / 112 with one warp, 23 / 23 with one CTA of
// 16 warps, 14 / 15 with 64 warps of 8 CTAs; 850 atoms in molecules 17 / 22 with one, 20 / 18 with two.  The largest power of two with which all atoms are resident at 16
// warps per SM (128 registers a thread).  Not with FAST, whose rows are those of large batches.
static Team team_of(const Work& w, bool fast)
{
    Team tm{1, 1};
    if (fast || w.N >= kSplitAtoms) return tm;
    int n = 2;
    while (n < kTeamMax * kTeamCtas && 2 * n * w.N <= (int64_t)16 * sm_count()) n *= 2;
    tm.warps = std::min(n, kTeamMax);
    tm.ctas = n / tm.warps;
    return tm;
}

bool desc_mma_fits(const Work& w, const DescDev& d, bool fast)
{
    return d.ang_kind == 0 && desc_smem(w, d, fast) <= kMaxSmem;
}

// four copies of the entries' sums when five CTAs per SM still fit, else fewer
static int adj_copies(const Work& w, const DescDev& d, bool fast)
{
    int nc = 4;
    while (nc > 1 && (size_t)adj_mma_smem(d, w.cap, nc, adj_fast(d, fast)).total(1) * kMW > 44 * 1024) nc /= 2;
    return nc;
}

// one shell chunk and at most two sector chunks: the block's gradient tile stays in registers
bool adj_mma_fits(const Work& w, const DescDev& d, bool fast)
{
    return d.ang_kind == 0 && d.n_ang_r <= 8 && d.n_theta <= 16 &&
           (size_t)kMW * adj_mma_smem(d, w.cap, 1, adj_fast(d, fast)).total(1) <= kMaxSmem;
}

cudaError_t launch_desc_mma(const Work& w, const DescDev& d, const int32_t* row_map, float* G_rows,
                            __nv_bfloat16* Gh, __nv_bfloat16* Gl, bool fast, cudaStream_t s)
{
    if (!desc_mma_fits(w, d, fast)) return cudaErrorNotSupported;
    if (w.N == 0) return cudaSuccess;
    const bool two = ((d.n_theta + 7) / 8) % 2 == 0;
    const int pw = log_terms(d, d.zeta);
    // pairs of bins on 8-byte boundaries; FP32 rows may be the caller's own, which start at any float
    const int even = ((d.D | d.rad_cols | d.n_ang_r) & 1) == 0 && (Gh || (reinterpret_cast<uintptr_t>(G_rows) & 7) == 0);
    const Team tm = team_of(w, desc_fast(d, fast));
    if (tm.warps > 1) {
        const size_t smem = desc_mma_atom_bytes<false>(w.cap) + tm.warps * desc_mma_warp_bytes<false>(two ? 2 : 1);
        auto run = [&](auto kern) { return launch_team(kern, w.N, tm, smem, s, d, w, row_map, G_rows, Gh, Gl, even); };
        if (pw == 8) return two ? run(k_desc_mma<false, 2, 8, true>) : run(k_desc_mma<false, 1, 8, true>);
        if (pw == 13) return two ? run(k_desc_mma<false, 2, 13, true>) : run(k_desc_mma<false, 1, 13, true>);
        return two ? run(k_desc_mma<false, 2, 0, true>) : run(k_desc_mma<false, 1, 0, true>);
    }
    const size_t smem = desc_smem(w, d, fast);
    auto run = [&](auto kern) { return launch_resident(kern, w.N, smem, s, d, w, row_map, G_rows, Gh, Gl, even); };
    if (desc_fast(d, fast)) return two ? run(k_desc_mma<true, 2, 0, false>) : run(k_desc_mma<true, 1, 0, false>);
    if (pw == 8) return two ? run(k_desc_mma<false, 2, 8, false>) : run(k_desc_mma<false, 1, 8, false>);
    if (pw == 13) return two ? run(k_desc_mma<false, 2, 13, false>) : run(k_desc_mma<false, 1, 13, false>);
    return two ? run(k_desc_mma<false, 2, 0, false>) : run(k_desc_mma<false, 1, 0, false>);
}

cudaError_t launch_adj_mma(const Work& w, const DescDev& d, const float* g_rows, float* F, float* vir_atom,
                           bool fast, cudaStream_t s)
{
    if (!adj_mma_fits(w, d, fast)) return cudaErrorNotSupported;
    if (w.N == 0) return cudaSuccess;
    const bool two = d.n_theta > 8;
    const int pw = log_terms(d, d.zeta - 1.f);
    int nc = adj_copies(w, d, fast);
    Team tm = team_of(w, adj_fast(d, fast));
    if (tm.warps > 1) {
        auto bytes = [&] { return (size_t)adj_mma_smem(d, w.cap, nc, false).total(tm.warps); };
        while (nc > 1 && bytes() > 100 * 1024) nc /= 2;
        while (tm.warps > 2 && bytes() > kMaxSmem) tm.warps /= 2;
        const size_t smem = bytes();
        auto run = [&](auto kern) { return launch_team(kern, w.N, tm, smem, s, d, w, g_rows, F, vir_atom, nc); };
        if (pw == 8) return two ? run(k_adj_mma<false, 2, 8, true>) : run(k_adj_mma<false, 1, 8, true>);
        if (pw == 13) return two ? run(k_adj_mma<false, 2, 13, true>) : run(k_adj_mma<false, 1, 13, true>);
        return two ? run(k_adj_mma<false, 2, 0, true>) : run(k_adj_mma<false, 1, 0, true>);
    }
    const size_t smem = (size_t)adj_mma_smem(d, w.cap, nc, adj_fast(d, fast)).total(1) * kMW;
    auto run = [&](auto kern) {
        return launch_resident(kern, w.N, smem, s, d, w, g_rows, F, vir_atom, nc);
    };
    if (adj_fast(d, fast)) return two ? run(k_adj_mma<true, 2, 0, false>) : run(k_adj_mma<true, 1, 0, false>);
    if (pw == 8) return two ? run(k_adj_mma<false, 2, 8, false>) : run(k_adj_mma<false, 1, 8, false>);
    if (pw == 13) return two ? run(k_adj_mma<false, 2, 13, false>) : run(k_adj_mma<false, 1, 13, false>);
    return two ? run(k_adj_mma<false, 2, 0, false>) : run(k_adj_mma<false, 1, 0, false>);
}

int small_rows_variant(const Work& w, const DescDev& d)
{
    return w.N < kSplitAtoms && desc_mma_fits(w, d, false) ? 5 : 0;
}

// exponents as for the adjoint's fast form
bool jvp_mma_fits(const Work& w, const DescDev& d)
{
    return d.ang_kind == 0 && adj_fast(d, true) && kMW * jvp_mma_bytes(w.cap) <= kMaxSmem;
}

cudaError_t launch_jvp_mma(const Work& w, const DescDev& d, const float* u, float* wdot_rows, cudaStream_t s)
{
    if (!jvp_mma_fits(w, d)) return cudaErrorNotSupported;
    if (w.N == 0) return cudaSuccess;
    const size_t smem = kMW * jvp_mma_bytes(w.cap);
    if (((d.n_theta + 7) / 8) % 2 == 0) return launch_resident(k_jvp_mma<2>, w.N, smem, s, d, w, u, wdot_rows);
    return launch_resident(k_jvp_mma<1>, w.N, smem, s, d, w, u, wdot_rows);
}

}  // namespace panna
