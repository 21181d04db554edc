// Layer products of the FP32 networks on the tensor cores with the accuracy of FP32 dot products:
// C[rows, N] = op(A)[rows, K] op(B)[K, N], the interface of k_gemm (mlp.cu), for batches past the
// single-launch path of mlp_small.cu.
//
// What is different from k_gemm.  Its FMAs and its shared-memory reads (each load returns at most 128
// bytes a cycle to an SM, also when lanes share addresses) take the same number of cycles, so it stays
// below half of the FMA rate.  Here both operands are split into TF32 parts x = hi + lo (11 + 11 bits, what
// is dropped at most one bit of FP32's 24) while they pass through registers on their way to shared
// memory, and tcgen05.mma forms hi hi, hi lo and lo hi (lo lo is below 2^-22).  The operands are read as
// they are, row-major FP32: no copies, no transposed weights, no alignment beyond k_gemm's.
//
// Accuracy.  The tensor cores truncate when they add to an accumulator, so a sum along all of K there has
// an error that grows with K (measured: six times that of an FP32 dot product).  The hi hi products of a
// step of 32 k (forward: of 16) go to one of three accumulators in turn, which the warps then add to their
// FP32 sums rounded to nearest; the cross terms, 2^-11 of the size, keep one accumulator for all of K.  What
// the truncation within a step loses on average (kXLost) is added back with them.  Error against 64 bits,
// relative 2-norm (k_gemm in brackets): forward, random operands, K = 768 1.6e-7 (5.0e-7), 256 1.2e-7
// (2.9e-7), 128 1.1e-7 (2.0e-7); positive ones 1.0e-7 (3.7e-7) at 768, 6e-8 (1.7e-7) at 128; input gradient
// 1.1e-7 (1.45e-7) and 5e-8 (1.2e-7) at 128.  Atomic energies of the four systems of the tests: half of
// k_gemm's error.  Errors that all rows share add up in an energy: the bit that a weight's split loses is cut
// off in every other row tile and rounded up in the others, which takes what a column's rows have in common
// from 0.4e-7 to 0.13e-7 of z (positive activations), and the sums of 4,096 atomic energies of 80 networks
// from 2.1e-7 off (RMS, of the sum of sizes) to 1.0e-7 (0.8e-7).
//
// CTA: a 128-row tile of one species, its 128-column tiles in turn, in steps of 32 k.  Warps 8..15 fetch A
// and warps 16..23 B (one or two steps ahead, into registers, by rows or by columns) and split it into the
// three stages (128-byte rows, 128-byte swizzle); warp 24 issues the MMAs (M = 128, K = 8 each); warps 0..7
// add up the finished accumulators and write out finished tiles.  Every wait is bounded: on time-out the CTA sets
// PANNA_ERR_TIMEOUT, waits for what it issued, frees its TMEM and returns.
// Bound: the waits between the roles (a step takes about 1,700 cycles, its MMAs 768, issue is 50 % busy; one
// set of 16 warps for splitting and adding took 3,000).  Registers: the adders' sums must not spill, shared
// memory leaves the L1 no room for them (the forward product without 16-byte loads spills 12 bytes).
// Measured (17,396 rows, us; k_gemm -> here): K = 768, N = 128: 110 -> 48; K = 128, N = 32: 24 -> 16; input
// gradient K = 128, N = 768: 121 -> 48; tangent K = 768 (before: a pass that split the operand, then TMA and
// MMAs) 86 -> 51; weight gradient 768 x 128 (before: passes that transposed and split both operands) 163 -> 91.
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "mlp.cuh"
#include "tc.cuh"

namespace panna {

namespace {

constexpr int kXAdd = 8, kXSplit = 8;                  // warps that add up, that split each operand
constexpr int kXThreads = 32 * (kXAdd + 2 * kXSplit + 4);   // and one of four that issues the MMAs
// Registers a thread: 72 at launch (28 warps); 8 * 112 + 16 * 64 + 4 * 24 = 28 * 72
constexpr int kRegAdd = 112, kRegSplit = 64, kRegMma = 24;
template <int R> __device__ __forceinline__ void regs_up() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(R)); }
template <int R> __device__ __forceinline__ void regs_down() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(R)); }
constexpr int kXStages = 3, kXAcc = 3, kXK = 32;                  // k per stage: 128-byte rows
constexpr uint32_t kXTile = 128 * 128;                 // 128 rows of 32 floats
constexpr uint32_t kXStage = 4 * kXTile;               // A hi, A lo, B hi, B lo
constexpr int kXLd = 132;                              // row stride of a finished tile
constexpr uint32_t kXOut = 64 * kXLd * 4;              // half of it at a time
constexpr uint32_t kXCols = 512;                       // TMEM: kXAcc accumulators of hi hi, one of the cross terms
// What truncation takes from the sum of 32 k on average (0.75e-7 to 1.28e-7 by the signs of its products; of
// 16 k 0.44e-7 to 0.60e-7).  Energies add up over all atoms, so the forward product, where the rest of that
// bias would be seen, takes two accumulators of 16 k per step.
constexpr float kXLost = 1.0e-7f;
constexpr size_t kXSmem = 1024 + kXStages * kXStage + kXOut + 256;

__device__ __forceinline__ void mbar_arrive(uint64_t* bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// One lane of the warp (leader) issues.  The warp runs the loop around it as a whole, so that descriptors and
// indices stay in uniform registers: with the loop inside a branch of one lane an MMA took 150 cycles to issue.
__device__ __forceinline__ void mma_tf32(uint32_t leader, uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t acc)
{
    asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc), "r"(leader)
                 : "memory");
}

__device__ __forceinline__ uint32_t elect()
{
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p;
}

__device__ __forceinline__ float low_clear(float x) { return __uint_as_float(__float_as_uint(x) & 0xffffe000u); }

// x = hi + lo: hi rounded to TF32, lo the rest (at most 12 bits, of which TF32 keeps 11: the last one is cut off,
// or with up = kUp rounded up)
constexpr uint32_t kUp = 0x1000u;
__device__ __forceinline__ void split(float x, float& hi, float& lo, uint32_t up)
{
    hi = __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
    lo = __uint_as_float((__float_as_uint(x - hi) + up) & 0xffffe000u);
}

// the same where rounding would overflow, for infinities and NaN (x + x: a NaN that TF32 keeps as one)
__device__ __noinline__ float2 split_special(float x)
{
    if (!(fabsf(x) < __int_as_float(0x7f800000))) return make_float2(x + x, 0.f);
    const float h = low_clear(x);
    return make_float2(h, low_clear(x - h));
}

__device__ __forceinline__ void split4(float4 v, float4& h, float4& l, uint32_t up = 0u)
{
    split(v.x, h.x, l.x, up);
    split(v.y, h.y, l.y, up);
    split(v.z, h.z, l.z, up);
    split(v.w, h.w, l.w, up);
    float m;
    asm("{\n\t.reg .f32 a, b, c, d;\n\tabs.f32 a, %1;\n\tabs.f32 b, %2;\n\tabs.f32 c, %3;\n\tabs.f32 d, %4;\n\t"
        "max.NaN.f32 a, a, b;\n\tmax.NaN.f32 c, c, d;\n\tmax.NaN.f32 %0, a, c;\n\t}"
        : "=f"(m) : "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w));
    if (!(m < 3.3e38f)) {
        const float2 a = split_special(v.x), b = split_special(v.y), c = split_special(v.z), d = split_special(v.w);
        h = make_float4(a.x, b.x, c.x, d.x);
        l = make_float4(a.y, b.y, c.y, d.y);
    }
}

// 4 values of p, n of them existing (VEC: all or none, aligned).  Predicated and volatile: nothing touches
// the result until it is split, and the compiler does not move the loads down to there.
__device__ __forceinline__ float load1(const float* p, bool on)
{
    float v = 0.f;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p ld.global.f32 %0, [%1];\n\t}"
                 : "+f"(v) : "l"(p), "r"((int)on));
    return v;
}
template <bool VEC>
__device__ __forceinline__ float4 load4(const float* p, int n)
{
    if (!VEC) return make_float4(load1(p, n > 0), load1(p + 1, n > 1), load1(p + 2, n > 2), load1(p + 3, n > 3));
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.gt.s32 p, %5, 0;\n\t@p ld.global.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
                 : "+f"(v.x), "+f"(v.y), "+f"(v.z), "+f"(v.w) : "l"(p), "r"(n));
    return v;
}

// 32 columns of the warp's lanes
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
                 "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// The weight gradient's product (OP_WGRAD): sums over the atoms of an item (at most `chunk` atoms of one
// species; items in species order), C[m, n] = sum over r of Zb[r, m] A[r, n] + Zdb[r, m] Ad[r, n], m over
// the layer's outputs, n over its inputs; both operands are read by columns, first Zb and A in steps of 32
// atoms, then Zdb and Ad.  Column `ldb` of C is the bias, the sum of Zb.
struct WgradArgs {
    const float *B, *Bd;   // A, Ad
    int ldb, chunk;
};

// operand A by rows (with or without act') or columns, B by rows (W [N, K]) or columns (W [K, N])
enum { OP_ROWS = 0, OP_WGRAD = 1 };

template <bool B_TRANS, int PRO, int EPI, int OP, bool VEC>
__global__ void __launch_bounds__(kXThreads, 1)
k_gemm_x3(LayerArgs la, const float* __restrict__ theta, const int32_t* __restrict__ seg_off,
          const int32_t* __restrict__ tile_start, const float* __restrict__ A, int lda, const float* __restrict__ Zp,
          int ldp, float* __restrict__ C, int ldc, float* __restrict__ C2, const float* __restrict__ Ze, int lde,
          DevStatus* status, WgradArgs wg)
{
    constexpr int SUB = EPI == EPI_FWD ? 2 : 1, KS = 4 / SUB;   // accumulators per step, MMAs of each
    constexpr bool WG = OP == OP_WGRAD;   // A, Zp: Zb, Zdb; C: the items' parts
    extern __shared__ unsigned char smem_raw[];
    __shared__ float bias_part[WG ? 128 : 1];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    float* out = reinterpret_cast<float*>(smem + kXStages * kXStage);          // finished tile
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + kXStages * kXStage + kXOut);   // a stage's operands written
    uint64_t* empty = full + kXStages;   // and read by the MMAs
    uint64_t* accf = empty + kXStages;   // accumulator of a step complete
    uint64_t* acce = accf + kXAcc;       // and added up
    uint64_t* done = acce + kXAcc;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // work decode (whole-CTA returns happen before any barrier or TMEM use)
    int s = 0, r0, rend, k0 = 0, nk, nkh = 0;
    if (WG) {
        int item = blockIdx.x;
        for (;; ++s) {
            if (s == la.S) return;
            const int ni = (seg_off[s + 1] - seg_off[s] + wg.chunk - 1) / wg.chunk;
            if (item < ni) break;
            item -= ni;
        }
        k0 = seg_off[s] + item * wg.chunk;
        r0 = blockIdx.z * 128;
        rend = la.N[s];
        if (r0 >= rend) return;
        nkh = (min(wg.chunk, seg_off[s + 1] - k0) + kXK - 1) / kXK;
        nk = 2 * nkh;
        C += (size_t)blockIdx.x * lde * ldc;   // lde: rows of an item's part
    } else {
        const int tile = blockIdx.x;
        if (tile >= tile_start[la.S]) return;
        while (tile >= tile_start[s + 1]) ++s;
        r0 = seg_off[s] + (tile - tile_start[s]) * 128;
        rend = seg_off[s + 1];
        nk = (la.K[s] + kXK - 1) / kXK;
    }
    const int K = WG ? min(wg.chunk, seg_off[s + 1] - k0) : la.K[s], N = WG ? la.K[s] : la.N[s];
    if ((int)blockIdx.y * 128 >= N) return;
    const int tiles = ((N + 127) / 128 - (int)blockIdx.y + (int)gridDim.y - 1) / (int)gridDim.y;
    const int steps = tiles * nk;
    auto tile_n0 = [&](int t) { return ((int)blockIdx.y + t * (int)gridDim.y) * 128; };
    auto tile_bn = [&](int t) { return min(128, (N - tile_n0(t) + 15) & ~15); };

    if (tid == 0) {
        for (int i = 0; i < kXStages; ++i) { mbar_init(full + i, 2 * kXSplit); mbar_init(empty + i, 1); }
        for (int i = 0; i < kXAcc; ++i) { mbar_init(accf + i, 1); mbar_init(acce + i, kXAdd); }
        mbar_init(done, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    constexpr int kMmaWarp = kXAdd + 2 * kXSplit;
    if (warp == kMmaWarp) tmem_alloc(tmem_slot, kXCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    const float* W = WG ? nullptr : theta + la.w_off[s];

    if (warp >= kMmaWarp) {
        regs_down<kRegMma>();
        if (warp == kMmaWarp) {
            const uint32_t leader = elect();
            const uint32_t smem0 = smem_u32(smem);
            bool ok = true;
            for (int t = 0, x = 0; t < tiles && ok; ++t) {
                const uint32_t idesc = idesc_mma(true, 128, (uint32_t)tile_bn(t));
                for (int c = 0; c < nk; ++c, ++x) {
                    const int st = x % kXStages;
                    ok = __all_sync(0xffffffffu, mbar_wait(full + st, (uint32_t)(x / kXStages) & 1u, abort_flag));
                    // c == 0: the cross terms' accumulator is free once the tile before is added up
                    if (ok && x > 0 && c == 0) {
                        const int y = x * SUB - 1;
                        ok = __all_sync(0xffffffffu, mbar_wait(acce + y % kXAcc, (uint32_t)(y / kXAcc) & 1u, abort_flag));
                    }
                    if (!ok) break;
                    const uint64_t ah = sw128_desc(smem0 + st * kXStage), al = ah + (kXTile >> 4);
                    const uint64_t bh = ah + (2 * kXTile >> 4), bl = ah + (3 * kXTile >> 4);
                    const int ks = min(kXK, K - (WG && c >= nkh ? c - nkh : c) * kXK + 7) / 8;
#pragma unroll
                    for (int u = 0; u < SUB; ++u) {
                        const int y = x * SUB + u, b = y % kXAcc;
                        ok = ok && __all_sync(0xffffffffu, mbar_wait(acce + b, ((uint32_t)(y / kXAcc) & 1u) ^ 1u, abort_flag));
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int k = u * KS; k < (u + 1) * KS; ++k)   // 8 k are 32 bytes of a row
                            if (k < ks)
                                mma_tf32(leader, tmem + b * 128, ah + 2 * k, bh + 2 * k, idesc, k > u * KS ? 1u : 0u);
                        if (u == SUB - 1) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (k < ks) {
                                    mma_tf32(leader, tmem + kXAcc * 128, ah + 2 * k, bl + 2 * k, idesc, (c | k) ? 1u : 0u);
                                    mma_tf32(leader, tmem + kXAcc * 128, al + 2 * k, bh + 2 * k, idesc, 1u);
                                }
                            if (leader) tc_commit(empty + st);
                        }
                        if (leader) tc_commit(accf + b);
                    }
                    if (!ok) break;
                }
            }
            if (!ok) *abort_flag = 1;
            if (leader) tc_commit(done);
            __syncwarp();
            mbar_wait(done, 0, nullptr);   // no TMEM release under running MMAs
        }
    } else if (warp >= kXAdd) {
        // operand splitters; a time-out leaves their loop running with waits that fail at once
        regs_down<kRegSplit>();
        const bool is_b = warp >= kXAdd + kXSplit;
        const int w = (warp - kXAdd) % kXSplit, tw = w * 32 + lane;
        const int row = tw >> 3, kq = (tw & 7) * 4;                       // from rows: rows row + 32 i, k kq .. kq + 3
        // from columns: column nc, k 4 kc + 8 i .. + 3 (a warp's load is 128 bytes of a row of memory, and the
        // four values of a column are 16 bytes of a row of the stage)
        const int nc = (w & 3) * 32 + lane, kc = w >> 2;
        // 16-byte columns of a row are permuted by the row's number mod 8 (128-byte swizzle)
        const uint32_t off = row * 128 + (((tw & 7) ^ (row & 7)) << 4);
        auto run = [&](auto fetch, auto put) {
            // two steps ahead; with act' one (its Z takes the other step's registers)
            constexpr int D = PRO == PRO_DACT ? 1 : 2;
            float4 v[D][4], z[PRO == PRO_DACT ? 4 : 1];
            int ft = 0, fc = 0;   // tile and k step of the next fetch
            auto next = [&](float4 (&u)[4]) {
                fetch(u, z, tile_n0(ft), fc * kXK);
                if (++fc == nk) { fc = 0; ++ft; }
            };
            auto step = [&](int x, float4 (&u)[4]) {
                const int st = x % kXStages;
                if (mbar_wait(empty + st, ((uint32_t)(x / kXStages) & 1u) ^ 1u, abort_flag)) {
                    put(smem + st * kXStage, u, z);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) mbar_arrive(full + st);
                } else {
                    *abort_flag = 1;
                }
                if (x + D < steps) next(u);
            };
#pragma unroll
            for (int d = 0; d < D; ++d)
                if (d < steps) next(v[d]);
            for (int x = 0; x < steps; x += D)
#pragma unroll
                for (int d = 0; d < D; ++d)
                    if (x + d < steps) step(x + d, v[d]);
        };
        auto put_rows = [&](uint8_t* hi, uint8_t* lo, const float4 (&u)[4], uint32_t up = 0u) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 h, l;
                split4(u[i], h, l, up);
                *reinterpret_cast<float4*>(hi + off + i * 4096) = h;
                *reinterpret_cast<float4*>(lo + off + i * 4096) = l;
            }
        };
        auto put_cols = [&](uint8_t* hi, uint8_t* lo, const float4 (&u)[4]) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const uint32_t o = nc * 128 + (((kc + 2 * i) ^ (nc & 7)) << 4);
                float4 h, l;
                split4(u[i], h, l);
                *reinterpret_cast<float4*>(hi + o) = h;
                *reinterpret_cast<float4*>(lo + o) = l;
            }
        };
        // column nc (on: it exists) of the rows p, p + ld, ..., of which `rows` exist
        auto fetch_cols = [&](float4 (&u)[4], const float* p, int ld, int rows, bool on) {
            p += (size_t)(4 * kc) * ld + nc;
            rows = on ? rows - 4 * kc : 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                u[i].x = load1(p, 8 * i < rows);
                u[i].y = load1(p + ld, 8 * i + 1 < rows);
                u[i].z = load1(p + 2 * (size_t)ld, 8 * i + 2 < rows);
                u[i].w = load1(p + 3 * (size_t)ld, 8 * i + 3 < rows);
                p += 8 * (size_t)ld;
            }
        };
        // 32 atoms from k on (those of the second product follow the first's): rows of x or xd, columns c0 on
        auto fetch_atoms = [&](float4 (&u)[4], const float* x, const float* xd, int ld, int c0, int cols, int k) {
            const bool second = k >= nkh * kXK;
            const int kr = second ? k - nkh * kXK : k;
            fetch_cols(u, (second ? xd : x) + (size_t)(k0 + kr) * ld + c0, ld, K - kr, c0 + nc < cols);
        };
        if (WG && !is_b) {
            float sum = 0.f;
            int px = 0;
            run([&](float4 (&u)[4], auto&, int, int k) { fetch_atoms(u, A, Zp, lda, r0, rend, k); },
                [&](uint8_t* st, float4 (&u)[4], auto&) {
                    if (px++ < nkh) {
#pragma unroll
                        for (int i = 0; i < 4; ++i) sum += (u[i].x + u[i].y) + (u[i].z + u[i].w);
                    }
                    put_cols(st, st + kXTile, u);
                });
            // the bias: two warps hold parts of a column
            if (blockIdx.y == 0) {
                if (kc == 1) bias_part[nc] = sum;
                asm volatile("bar.sync 2, %0;" ::"r"(32 * kXSplit) : "memory");
                if (kc == 0 && r0 + nc < rend) C[(size_t)(r0 + nc) * ldc + wg.ldb] = sum + bias_part[nc];
            }
        } else if (WG) {
            run([&](float4 (&u)[4], auto&, int n0, int k) { fetch_atoms(u, wg.B, wg.Bd, wg.ldb, n0, N, k); },
                [&](uint8_t* st, float4 (&u)[4], auto&) { put_cols(st + 2 * kXTile, st + 3 * kXTile, u); });
        } else if (!is_b) {
            const float* Ar = A + (size_t)(r0 + row) * lda + kq;
            const float* Zr = PRO == PRO_DACT ? Zp + (size_t)(r0 + row) * ldp + kq : nullptr;
            const int pact = la.pact[s];
            run([&](float4 (&u)[4], auto& z, int, int k) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int left = r0 + row + 32 * i < rend ? K - k - kq : 0;
                    u[i] = load4<VEC>(Ar + (size_t)(32 * i) * lda + k, left);
                    if (PRO == PRO_DACT) z[i] = load4<VEC>(Zr + (size_t)(32 * i) * ldp + k, left);
                }
            }, [&](uint8_t* st, float4 (&u)[4], auto& z) {
                if (PRO == PRO_DACT) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        u[i].x *= act_d1(pact, z[i].x);
                        u[i].y *= act_d1(pact, z[i].y);
                        u[i].z *= act_d1(pact, z[i].z);
                        u[i].w *= act_d1(pact, z[i].w);
                    }
                }
                put_rows(st, st + kXTile, u);
            });
        } else if (B_TRANS) {
            // The bit that a weight loses is the same for all rows, and energies add up over them: every other row
            // tile rounds it up.
            const uint32_t up = EPI == EPI_FWD && (blockIdx.x & 1) ? kUp : 0u;
            auto rows_of_w = [&](auto vec) {
                run([&](float4 (&u)[4], auto&, int n0, int k) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int n = n0 + row + 32 * i;
                        u[i] = load4<decltype(vec)::value>(W + (size_t)n * K + k + kq, n < N ? K - k - kq : 0);
                    }
                }, [&](uint8_t* st, float4 (&u)[4], auto&) { put_rows(st + 2 * kXTile, st + 3 * kXTile, u, up); });
            };
            // a species' weights start anywhere in theta
            if ((reinterpret_cast<uintptr_t>(W) & 15) == 0 && (K & 3) == 0) rows_of_w(std::true_type{});
            else rows_of_w(std::false_type{});
        } else {
            run([&](float4 (&u)[4], auto&, int n0, int k) { fetch_cols(u, W + (size_t)k * N + n0, N, K - k, n0 + nc < N); },
                [&](uint8_t* st, float4 (&u)[4], auto&) { put_cols(st + 2 * kXTile, st + 3 * kXTile, u); });
        }
    } else {
        regs_up<kRegAdd>();
        // sums of this warp's quarter of the rows (TMEM lanes: warp mod 4) and half of the columns
        const int q = warp & 3, c0 = (warp >> 2) * 64;
        const uint32_t lanes = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
        float acc[64];
        auto add = [&](uint32_t col) {
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                float v[32];
                tc_ld32(lanes + col + 32 * x, v);
#pragma unroll
                for (int j = 0; j < 32; ++j) acc[32 * x + j] += v[j];
            }
        };
        // an infinite operand leaves its products in the sum of hi hi, and 0 times infinity in the cross terms
        auto add_cross = [&](uint32_t col, float lost) {
#pragma unroll
            for (int x = 0; x < 2; ++x) {
                float v[32];
                tc_ld32(lanes + col + 32 * x, v);
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const float a = acc[32 * x + j];
                    if (fabsf(a) < __int_as_float(0x7f800000)) acc[32 * x + j] = a + fmaf(lost, a, v[j]);
                }
            }
        };
        const float* bias = WG ? nullptr : theta + la.b_off[s];
        const bool vst = ((reinterpret_cast<uintptr_t>(C) & 15) == 0) && (ldc & 3) == 0 &&
                         (EPI == EPI_STORE || ((reinterpret_cast<uintptr_t>(C2) & 15) == 0));
        // a finished tile through shared memory, 64 rows at a time: its rows then leave as contiguous float4.
        // Not unrolled: this code runs once or a few times per CTA, and fetching it is what it takes.
        auto finish = [&](int t) {
            const int nb4 = tile_n0(t) + lane * 4, act = la.act[s];
            float bv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) bv[j] = EPI == EPI_FWD && nb4 + j < N ? bias[nb4 + j] : 0.f;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                if ((q >> 1) == h) {
                    float4* dst = reinterpret_cast<float4*>(out + ((q & 1) * 32 + lane) * kXLd + c0);
#pragma unroll
                    for (int j = 0; j < 16; ++j)
                        dst[j] = make_float4(acc[4 * j], acc[4 * j + 1], acc[4 * j + 2], acc[4 * j + 3]);
                }
                asm volatile("bar.sync 1, %0;" ::"r"(32 * kXAdd) : "memory");
                const int rows = min(64, rend - r0 - 64 * h);
#pragma unroll (EPI == EPI_TAN ? 2 : 1)
                for (int rr = warp; rr < rows; rr += kXAdd) {
                    const int r = r0 + 64 * h + rr;
                    if (nb4 >= N) break;
                    const float4 t4 = *reinterpret_cast<const float4*>(out + rr * kXLd + lane * 4);
                    float v[4] = {t4.x, t4.y, t4.z, t4.w}, v2[4], ze[4];
                    float* c = C + (size_t)r * ldc + nb4;
                    float* c2 = EPI == EPI_STORE ? nullptr : C2 + (size_t)r * ldc + nb4;
                    const int nv = min(4, N - nb4);
                    if (EPI == EPI_TAN) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) ze[j] = j < nv ? Ze[(size_t)r * lde + nb4 + j] : 0.f;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (EPI == EPI_FWD) {
                            v[j] += bv[j];
                            v2[j] = act_f(act, v[j]);
                        } else if (EPI == EPI_TAN) {
                            v2[j] = act_d1(act, ze[j]) * v[j];
                        }
                    }
                    if (vst && nv == 4) {
                        *reinterpret_cast<float4*>(c) = make_float4(v[0], v[1], v[2], v[3]);
                        if (EPI != EPI_STORE) *reinterpret_cast<float4*>(c2) = make_float4(v2[0], v2[1], v2[2], v2[3]);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (j >= nv) break;
                            c[j] = v[j];
                            if (EPI != EPI_STORE) c2[j] = v2[j];
                        }
                    }
                }
                asm volatile("bar.sync 1, %0;" ::"r"(32 * kXAdd) : "memory");
            }
        };
        // After a time-out the warps go on through all steps (their waits then fail at once), so that they
        // meet at every barrier, and agree before a tile is finished.
        int dt = 0, dc = 0;   // tile and part of it (SUB per k step) of the next drain
        auto drain = [&](int y) {
            const int b = y % kXAcc;
            const bool ok = mbar_wait(accf + b, (uint32_t)(y / kXAcc) & 1u, abort_flag);
            if (ok) {
                tc_fence_after();
                if (dc == 0) {
#pragma unroll
                    for (int j = 0; j < 64; ++j) acc[j] = 0.f;
                }
                const bool used = c0 < tile_bn(dt);
                // the last step may be too short for its second part
                if (used && (SUB == 1 || dc * KS * 8 < K)) add((uint32_t)b * 128);
                if (dc == nk * SUB - 1 && used) add_cross(kXAcc * 128, kXLost / SUB);
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(acce + b);
            } else {
                *abort_flag = 1;
            }
            if (++dc < nk * SUB) return;
            dc = 0;
            uint32_t bad;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\tbarrier.cta.red.or.pred p, 1, %2, p;\n\t"
                         "selp.u32 %0, 1, 0, p;\n\t}"
                         : "=r"(bad) : "r"(*abort_flag), "r"(32 * kXAdd) : "memory");
            if (!bad) finish(dt);
            ++dt;
        };
        for (int y = 0; y < steps * SUB; ++y) drain(y);
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *abort_flag) set_status(status, PANNA_ERR_TIMEOUT, blockIdx.x);
    if (warp == kMmaWarp) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem, kXCols);
    }
}

}  // namespace

template <bool B_TRANS, int PRO, int EPI>
cudaError_t launch_gemm_x3(dim3 grid, cudaStream_t s, const LayerArgs& la, const float* theta, const int32_t* seg_off,
                           const int32_t* tile_start, const float* A, int lda, const float* Zp, int ldp, float* C,
                           int ldc, float* C2, const float* Ze, int lde, DevStatus* status)
{
    // 16-byte loads need aligned rows of A and Z
    auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
    bool vec = aligned(A) && lda % 4 == 0 && (PRO == PRO_NONE || (aligned(Zp) && ldp % 4 == 0));
    for (int q = 0; q < la.S; ++q) vec = vec && la.K[q] % 4 == 0;
    auto kern = vec ? k_gemm_x3<B_TRANS, PRO, EPI, OP_ROWS, true> : k_gemm_x3<B_TRANS, PRO, EPI, OP_ROWS, false>;
    cudaError_t e = allow_smem(kern, kXSmem);
    if (e != cudaSuccess) return e;
    kern<<<grid, kXThreads, kXSmem, s>>>(la, theta, seg_off, tile_start, A, lda, Zp, ldp, C, ldc, C2, Ze, lde, status,
                                         WgradArgs{});
    return cudaGetLastError();
}

#define PANNA_X3(BT, PRO, EPI)                                                                                     \
    template cudaError_t launch_gemm_x3<BT, PRO, EPI>(dim3, cudaStream_t, const LayerArgs&, const float*,          \
                                                      const int32_t*, const int32_t*, const float*, int,           \
                                                      const float*, int, float*, int, float*, const float*, int,   \
                                                      DevStatus*);
PANNA_X3(true, PRO_NONE, EPI_FWD)
PANNA_X3(true, PRO_NONE, EPI_TAN)
PANNA_X3(false, PRO_DACT, EPI_STORE)
PANNA_X3(false, PRO_NONE, EPI_STORE)
#undef PANNA_X3

// ------------------------------------------------------------------ weight gradient of the FP32 networks

namespace {

// the species of an item (up to `chunk` atoms of one species, items in species order) and its first item
__device__ __forceinline__ bool item_species(int S, const int32_t* __restrict__ seg_off, int chunk, int item, int& s,
                                             int& first)
{
    for (s = 0, first = 0; s < S; ++s) {
        const int ni = (seg_off[s + 1] - seg_off[s] + chunk - 1) / chunk;
        if (item < first + ni) return true;
        first += ni;
    }
    return false;
}

// Weight gradient of a narrow layer (M x (K+1) <= 8192 outputs) straight from the row-major
// adjoints Zb, Zdb [rows, M] and inputs A, Ad [rows, K]: one CTA per (item = species chunk of
// atoms, split of that chunk); every thread owns up to 32 outputs o = m (K+1) + n (n == K: the
// bias), rows pass through shared memory 32 at a time.  The partial of (item, split) goes to
// part[(item * splits + split) * M (K+1) + o], so item order stays the reduction order.
constexpr int kSmallRows = 32, kSmallOut = 32;
__global__ void __launch_bounds__(256)
k_wgrad_small(int S, const int32_t* __restrict__ seg_off, int chunk,
              int splits, int M, int K, const float* __restrict__ Zb, const float* __restrict__ Zdb,
              const float* __restrict__ A, const float* __restrict__ Ad, float* __restrict__ part)
{
    extern __shared__ float sh[];
    const int item = blockIdx.x;
    int s = 0, first = 0;
    if (!item_species(S, seg_off, chunk, item, s, first)) return;
    const int per = (chunk / splits + kSmallRows - 1) / kSmallRows * kSmallRows;
    const int c0 = (item - first) * chunk + blockIdx.y * per;
    const int cend = min((item - first + 1) * chunk, c0 + per);
    const int cnt = seg_off[s + 1] - seg_off[s];
    const int a0 = seg_off[s] + min(cnt, c0), a1 = seg_off[s] + min(cnt, cend);
    float* sZ = sh;
    float* sZd = sZ + kSmallRows * M;
    float* sA = sZd + kSmallRows * M;
    float* sAd = sA + kSmallRows * K;
    const int O = M * (K + 1);
    const int tid = threadIdx.x;
    float acc[kSmallOut];
#pragma unroll
    for (int j = 0; j < kSmallOut; ++j) acc[j] = 0.f;
    for (int r0 = a0; r0 < a1; r0 += kSmallRows) {
        const int nr = min(kSmallRows, a1 - r0);
        __syncthreads();
        for (int idx = tid; idx < kSmallRows * M; idx += 256) {
            const int rr = idx / M;
            sZ[idx] = rr < nr ? Zb[(size_t)r0 * M + idx] : 0.f;
            sZd[idx] = rr < nr ? Zdb[(size_t)r0 * M + idx] : 0.f;
        }
        for (int idx = tid; idx < kSmallRows * K; idx += 256) {
            const int rr = idx / K;
            sA[idx] = rr < nr ? A[(size_t)r0 * K + idx] : 0.f;
            sAd[idx] = rr < nr ? Ad[(size_t)r0 * K + idx] : 0.f;
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < kSmallOut; ++j) {
            const int o = j * 256 + tid;
            if (o >= O) break;
            const int m = o / (K + 1), n = o % (K + 1);
            float a = acc[j];
            if (n < K) {
                for (int rr = 0; rr < kSmallRows; ++rr)
                    a = fmaf(sZ[rr * M + m], sA[rr * K + n], fmaf(sZd[rr * M + m], sAd[rr * K + n], a));
            } else {
                for (int rr = 0; rr < kSmallRows; ++rr) a += sZ[rr * M + m];
            }
            acc[j] = a;
        }
    }
    float* out = part + ((size_t)item * splits + blockIdx.y) * O;
#pragma unroll
    for (int j = 0; j < kSmallOut; ++j) {
        const int o = j * 256 + tid;
        if (o >= O) break;
        out[o] = acc[j];
    }
}

// The same partial sums with 4 x 4 register blocks (M and K multiples of 4, (M/4)(K/4) <= 256
// blocks): thread b owns weights m in [4 (b / (K/4)), +4), n in [4 (b % (K/4)), +4), and the
// threads of the first n block also the 4 biases; per staged row it reads 4 + 4 float4 from
// shared memory for 32 FMAs (the scalar kernel above reads 4 floats per 2 FMAs).
__global__ void __launch_bounds__(256)
k_wgrad_small4(int S, const int32_t* __restrict__ seg_off, int chunk,
               int splits, int M, int K, const float* __restrict__ Zb, const float* __restrict__ Zdb,
               const float* __restrict__ A, const float* __restrict__ Ad, float* __restrict__ part)
{
    extern __shared__ __align__(16) float sh4[];
    const int item = blockIdx.x;
    int s = 0, first = 0;
    if (!item_species(S, seg_off, chunk, item, s, first)) return;
    const int per = (chunk / splits + kSmallRows - 1) / kSmallRows * kSmallRows;
    const int c0 = (item - first) * chunk + blockIdx.y * per;
    const int cend = min((item - first + 1) * chunk, c0 + per);
    const int cnt = seg_off[s + 1] - seg_off[s];
    const int a0 = seg_off[s] + min(cnt, c0), a1 = seg_off[s] + min(cnt, cend);
    float* sZ = sh4;
    float* sZd = sZ + kSmallRows * M;
    float* sA = sZd + kSmallRows * M;
    float* sAd = sA + kSmallRows * K;
    const int tid = threadIdx.x;
    const int K4 = K >> 2, nblk = (M >> 2) * K4;
    const bool own = tid < nblk;
    const int m0 = own ? (tid / K4) * 4 : 0, n0 = own ? (tid % K4) * 4 : 0;
    float acc[4][4], bias[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
        bias[a] = 0.f;
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
    }
    for (int r0 = a0; r0 < a1; r0 += kSmallRows) {
        const int nr = min(kSmallRows, a1 - r0);
        __syncthreads();
        for (int idx = tid; idx < kSmallRows * M; idx += 256) {
            const int rr = idx / M;
            sZ[idx] = rr < nr ? Zb[(size_t)r0 * M + idx] : 0.f;
            sZd[idx] = rr < nr ? Zdb[(size_t)r0 * M + idx] : 0.f;
        }
        for (int idx = tid; idx < kSmallRows * K; idx += 256) {
            const int rr = idx / K;
            sA[idx] = rr < nr ? A[(size_t)r0 * K + idx] : 0.f;
            sAd[idx] = rr < nr ? Ad[(size_t)r0 * K + idx] : 0.f;
        }
        __syncthreads();
        if (own) {
            for (int rr = 0; rr < kSmallRows; ++rr) {
                const float4 z = *reinterpret_cast<const float4*>(sZ + rr * M + m0);
                const float4 zd = *reinterpret_cast<const float4*>(sZd + rr * M + m0);
                const float4 a = *reinterpret_cast<const float4*>(sA + rr * K + n0);
                const float4 ad = *reinterpret_cast<const float4*>(sAd + rr * K + n0);
                const float zv[4] = {z.x, z.y, z.z, z.w}, zdv[4] = {zd.x, zd.y, zd.z, zd.w};
                const float av[4] = {a.x, a.y, a.z, a.w}, adv[4] = {ad.x, ad.y, ad.z, ad.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    bias[i] += zv[i];
#pragma unroll
                    for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(zv[i], av[j], fmaf(zdv[i], adv[j], acc[i][j]));
                }
            }
        }
    }
    if (!own) return;
    float* out = part + ((size_t)item * splits + blockIdx.y) * ((size_t)M * (K + 1));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int j = 0; j < 4; ++j) out[(size_t)(m0 + i) * (K + 1) + n0 + j] = acc[i][j];
        if (n0 == 0) out[(size_t)(m0 + i) * (K + 1) + K] = bias[i];
    }
}

// dtheta of one layer from the per-item partial sums (splits per item): n < K_s: weight W[m][n]; n ==
// bias_col: bias b[m].  CTA: 256 / WAYS outputs, the parts dealt to WAYS threads each, whose sums are added
// in order.  Narrow layers have many parts: with one thread per output, a chain of 300 loads, 1024
// molecules' 32 x 129 layer took 15 us, with eight 7; wide ones few: 8.5 us with one, 27 with eight.
template <int WAYS>
__global__ void __launch_bounds__(256)
k_wgrad_reduce(LayerArgs la, const int32_t* __restrict__ seg_off, int chunk, int splits, int Mvalid, int ldn,
               int bias_col, const float* __restrict__ part, float* __restrict__ dtheta)
{
    constexpr int OUT = 256 / WAYS;
    __shared__ float sums[WAYS][OUT];
    const int x = threadIdx.x % OUT, y = threadIdx.x / OUT;
    const int64_t idx = (int64_t)blockIdx.x * OUT + x;
    const int s = (int)(idx / ((int64_t)Mvalid * ldn));
    const int m = (int)((idx / ldn) % Mvalid);
    const int n = (int)(idx % ldn);
    const bool on = s < la.S && m < la.N[s] && (n < la.K[s] || n == bias_col);
    float acc = 0.f;
    if (on) {
        int it = 0;
        for (int q = 0; q < s; ++q) it += (seg_off[q + 1] - seg_off[q] + chunk - 1) / chunk;
        const int end = (it + (seg_off[s + 1] - seg_off[s] + chunk - 1) / chunk) * splits;
        for (it = it * splits + y; it < end; it += WAYS) acc += part[((size_t)it * Mvalid + m) * ldn + n];
    }
    if (WAYS > 1) {
        sums[y][x] = acc;
        __syncthreads();
        if (y) return;
#pragma unroll
        for (int w = 1; w < WAYS; ++w) acc += sums[w][x];
    }
    if (!on) return;
    if (n < la.K[s]) dtheta[la.w_off[s] + (int64_t)m * la.K[s] + n] = acc;
    else dtheta[la.b_off[s] + m] = acc;
}

// How a layer's weight gradient is summed: on the CUDA cores when it is narrow (rows of its inputs and
// adjoints in 48 KB of shared memory), else by k_gemm_x3 with as many items as fill the SMs once, no
// shorter than 256 atoms (each leaves a part to add up).
struct WgradPlan {
    bool narrow;
    int chunk, items, splits, ldn;
    size_t floats;   // of the parts
};

WgradPlan wgrad_plan(const MlpPlan& p, int64_t N, int l)
{
    const int K = p.ld[l], M = p.ld[l + 1], O = M * (K + 1);
    WgradPlan w{};
    w.narrow = l > 0 && O <= 256 * kSmallOut && M + K <= 192;
    if (w.narrow) {
        w.chunk = (int)std::max<int64_t>(512, (N / 256 + 31) / 32 * 32);
        size_t wide = 0;
        for (int q = 0; q < p.L; ++q) wide = std::max(wide, (size_t)p.ld[q + 1] * (p.ld[q] + 1));
        w.splits = (int)std::max<size_t>(1, std::min<size_t>(8, wide / O));
        w.ldn = K + 1;
    } else {
        const int64_t tiles = (int64_t)((K + 127) / 128) * ((M + 127) / 128);
        const int64_t items = std::max<int64_t>(1, sm_count() / tiles - p.S);
        w.chunk = (int)std::max<int64_t>(256, ((N + items - 1) / items + 31) / 32 * 32);
        w.splits = 1;
        w.ldn = (K + 4) & ~3;   // K weights, the bias
    }
    w.items = (int)((N + w.chunk - 1) / w.chunk) + p.S;
    w.floats = (size_t)w.items * w.splits * M * w.ldn;
    return w;
}

}  // namespace

size_t wgrad_workspace_bytes(const MlpPlan& p, int64_t N)
{
    size_t f = 0;
    for (int l = 0; l < p.L; ++l) f = std::max(f, wgrad_plan(p, N, l).floats);
    return f * sizeof(float);
}

cudaError_t wgrad_layer(const MlpPlan& p, const MlpBuffers& b, int64_t N, float* part, int l, const LayerArgs& la,
                        const float* A, const float* Ad, float* dtheta, cudaStream_t s, int* launches)
{
    const WgradPlan w = wgrad_plan(p, N, l);
    const int K = p.ld[l], M = p.ld[l + 1];
    if (w.narrow) {
        const size_t smem = (size_t)kSmallRows * 2 * (M + K) * sizeof(float);
        dim3 grid((unsigned)w.items, (unsigned)w.splits);
        if (M % 4 == 0 && K % 4 == 0 && (M / 4) * (K / 4) <= 256)
            k_wgrad_small4<<<grid, 256, smem, s>>>(p.S, b.seg_off, w.chunk, w.splits, M, K, b.Zb, b.Zdb, A, Ad, part);
        else
            k_wgrad_small<<<grid, 256, smem, s>>>(p.S, b.seg_off, w.chunk, w.splits, M, K, b.Zb, b.Zdb, A, Ad, part);
    } else {
        auto kern = k_gemm_x3<false, PRO_NONE, EPI_STORE, OP_WGRAD, false>;
        cudaError_t e = allow_smem(kern, kXSmem);
        if (e != cudaSuccess) return e;
        dim3 grid((unsigned)w.items, (unsigned)((K + 127) / 128), (unsigned)((M + 127) / 128));
        kern<<<grid, kXThreads, kXSmem, s>>>(la, nullptr, b.seg_off, nullptr, b.Zb, M, b.Zdb, M, part, w.ldn, nullptr,
                                             nullptr, M, b.status, WgradArgs{A, Ad, K, w.chunk});
    }
    const int64_t n = (int64_t)p.S * M * w.ldn;
    if (w.narrow)
        k_wgrad_reduce<8><<<(unsigned)((n + 31) / 32), 256, 0, s>>>(la, b.seg_off, w.chunk, w.splits, M, w.ldn, K, part,
                                                                    dtheta);
    else
        k_wgrad_reduce<1><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(la, b.seg_off, w.chunk, w.splits, M, w.ldn, K, part,
                                                                      dtheta);
    *launches += 2;
    return cudaGetLastError();
}

}  // namespace panna
