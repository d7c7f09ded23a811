// Dense hypothesis scoring: for every P3P hypothesis h of frame t,
//   L_h = sum_j W_t^j log[rho_j(h) / (rho_j(h) + mu_j)]
// over the pixels whose pi_{t-1} is valid -- the MIE criterion of Eq. 10 with
// the pose as the free variable (Eq. 9's MLE form as the ablation variant).
//
// Per (hypothesis, pixel) pair, with the scaled form (E, tt) of the hypothesis
// and the pixel's normalised coordinates, inverse depth and flow over fx:
//   a_z, U, V               three contractions (score_ops.cuh)
//   r_u  = U / (1 + a_z), r_v = V / (1 + a_z)          (residual / fx)
//   xs   = r_u^2 + r_v^2, clamped to [xs_min, xs_max]  (squared residual / fx^2)
//   s    = beta log2(xs) + beta_k               (log2 of (x/alpha)^beta)
//   r    = Cp xs (2^s + 2 + 2^-s)               (= mu / rho, Eqs. 3-4, 7)
//   ell  = -log1p(r); behind camera t (1 + a_z <= 0) rho := mu, ell = -log 2.
// The contractions run on the tensor cores (tcgen05, BF16 slices, FP32
// accumulation in tensor memory); the rest is FP32 on packed pairs of
// hypotheses (.f32x2), with the SFU's rcp, lg2 and ex2.
#include <cmath>
#include <mutex>
#include <type_traits>
#include <vector>

#include <algorithm>

#include "score_ops.cuh"
#include "tc.cuh"
#include "voldor_internal.cuh"

namespace vd {

__device__ __forceinline__ float mufu_rcp(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float mufu_lg2(float x)
{
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float mufu_ex2(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

struct HypF {
    float e0, e1, e2, e3, e4, e5, e6, e7, e8, t0, t1, t2;
};

// log2(1 + r) for r >= 0: below 1/8 r * P(r) with P the degree-3 Chebyshev
// interpolant of log2(1 + r)/r on [0, 1/8] (coefficients highest degree first;
// relative error at most 4.2e-7 in FP32 Horner form, mean 1.9e-7: the nearest
// singularity, r = -1, is seventeen half-widths from the interval, so each
// degree gains a factor ~34); above, lg2(1 + r), an absolute-accuracy
// approximation whose result there is at least log2(9/8) = 0.17. Against the
// earlier degree-4 interpolant on [0, 1/4] this saves one FMA per pair and
// moved the driving window's dense scores by at most 3.1e-8 relative.
constexpr float kL1pC3 = -2.977027297e-01f, kL1pC2 = 4.761879444e-01f, kL1pC1 = -7.212317586e-01f,
                kL1pC0 = 1.442694545e+00f;
constexpr float kL1pMax = 0.125f;

__device__ __forceinline__ float log2_1p_pos(float r)
{
    float s = fmaf(r, kL1pC3, kL1pC2);
    s = fmaf(r, s, kL1pC1);
    s = fmaf(r, s, kL1pC0);
    const float small = r * s;
    const float big = mufu_lg2(1.f + r);
    return r < kL1pMax ? small : big;
}

// Scalar pair term of the allocation-free entry point: -ell / ln2 = log2(1 + mu/rho)
// of one (hypothesis, pixel) pair (MIE, Eq. 10), the projection in FP32 and a
// reciprocal to each pair; behind camera t (1 + a_z <= 0) rho := mu (r = 1).
__device__ __forceinline__ float pair_term2(const HypF& h, const float4 a, const float4 b, float xs_min, float xs_max)
{
    const float xb = a.x, yb2 = a.y, w = a.z, ut = a.w;
    const float vt = b.x, beta = b.y, beta_k = b.z, Cp = b.w;
    const float ax = fmaf(h.e0, xb, fmaf(h.e1, yb2, fmaf(h.t0, w, h.e2)));
    const float ay = fmaf(h.e3, xb, fmaf(h.e4, yb2, fmaf(h.t1, w, h.e5)));
    const float az = fmaf(h.e6, xb, fmaf(h.e7, yb2, fmaf(h.t2, w, h.e8)));
    const float den = 1.f + az;
    const float rd = mufu_rcp(den);
    const float ru = fmaf(fmaf(-xb, az, ax), rd, -ut);
    const float rv = fmaf(fmaf(-yb2, az, ay), rd, -vt);
    const float xs = fminf(fmaxf(fmaf(ru, ru, rv * rv), xs_min), xs_max);
    const float sg = fabsf(fmaf(beta, mufu_lg2(xs), beta_k));
    const float r = Cp * xs * (mufu_ex2(sg) + (2.f + mufu_ex2(-sg)));
    return den > 0.f ? log2_1p_pos(r) : 1.f;
}

// ---------------------------------------------------------------------------
// Packed pair arithmetic (.f32x2).
// ---------------------------------------------------------------------------
typedef unsigned long long f2;      // {lo, hi} FP32 lanes

__device__ __forceinline__ f2 f2_pack(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}

__device__ __forceinline__ float f2_lo(f2 v)
{
    float lo;
    asm("mov.b64 {%0, _}, %1;" : "=f"(lo) : "l"(v));
    return lo;
}

__device__ __forceinline__ float f2_hi(f2 v)
{
    float hi;
    asm("mov.b64 {_, %0}, %1;" : "=f"(hi) : "l"(v));
    return hi;
}

__device__ __forceinline__ f2 f2_both(float v) { return f2_pack(v, v); }

__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f2 f2_sub(f2 a, f2 b)
{
    f2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ f2 f2_lg2(f2 v) { return f2_pack(mufu_lg2(f2_lo(v)), mufu_lg2(f2_hi(v))); }

// ---------------------------------------------------------------------------
// Terms of P hypothesis pairs against the lane's pixel, added to acc.
// ---------------------------------------------------------------------------
struct PixConst {
    f2 beta, beta_k, Cp, wq;         // Gaussian: Cp is the pixel's U0
    float xmu;                       // x_mu / fx^2: the squared residual at which rho = mu; Gaussian: V0
};

// The polynomial of log2_1p_pos for r < 1/8.
__device__ __forceinline__ f2 log2_1p_small(f2 r)
{
    f2 p = f2_fma(r, f2_both(kL1pC3), f2_both(kL1pC2));
    p = f2_fma(r, p, f2_both(kL1pC1));
    p = f2_fma(r, p, f2_both(kL1pC0));
    return f2_mul(r, p);
}

// log2(1 + r) from that polynomial (`small`) or, for r >= 1/8, lg2 of r1 = 1 + r; the
// lg2 is predicated, so a warp whose 32 pixels all lie below issues none.
__device__ __forceinline__ float lg2_if_large(float small, float r, float r1)
{
    static_assert(kL1pMax == 0.125f, "the literal below");
    asm("{\n .reg .pred p;\n setp.ge.f32 p, %1, 0f3E000000;\n @p lg2.approx.ftz.f32 %0, %2;\n}"
        : "+f"(small) : "f"(r), "f"(r1));
    return small;
}

// U, V and a_z of P pairs against the lane's pixel. One reciprocal serves the two
// lanes of a pair, 1 / d0 = d1 / (d0 d1), d = 1 + a_z: a nonzero d is at least 2^-25
// in size (the spacing of a_z near -1), so adding 2^-40 moves no d beyond its own
// rounding and keeps an exact 0 from spoiling its partner; above, kWild frames (the
// only ones where |d| may reach 2^62) take a reciprocal per lane. So does the Gaussian
// model, whose terms grow with the squared residual itself and carry every rounding of
// it, and it adds U0 and V0 here, rounded, instead of in the tensor core, which
// truncates: the error of its scores near the current pose, rms over 60 sets of
// hypotheses against 64 bits, is 0.99 of what it was with the projection in FP32, 1.17
// without the two. Behind the camera (d <= 0) rho := mu. The loops over P keep P independent chains side by
// side for the in-order issue.
template <int P, bool kMLE, bool kGauss, bool kWild>
__device__ __forceinline__ void score_pairs(const uint32_t* U, const uint32_t* V, const uint32_t* Z, const PixConst& q,
                                            float xs_min, float xs_max, f2* acc)
{
    auto at = [](const uint32_t* v, int i) { return f2_pack(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1])); };
    f2 nden[P];                                           // -(1 + a_z)
#pragma unroll
    for (int i = 0; i < P; ++i) nden[i] = f2_sub(f2_both(-1.f), at(Z, i));
    f2 xs[P], s[P], v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        f2 rd;                                            // -1 / (1 + a_z): squared below
        if (kWild || kGauss) {
            rd = f2_pack(mufu_rcp(f2_lo(nden[i])), mufu_rcp(f2_hi(nden[i])));
        } else {
            const f2 d = f2_add(nden[i], f2_both(9.094947e-13f));
            const float inv = mufu_rcp(f2_lo(d) * f2_hi(d));
            rd = f2_pack(inv * f2_hi(d), inv * f2_lo(d));
        }
        const f2 u = kGauss ? f2_add(at(U, i), q.Cp) : at(U, i), w = kGauss ? f2_add(at(V, i), f2_both(q.xmu)) : at(V, i);
        const f2 ru = f2_mul(u, rd), rv = f2_mul(w, rd);
        const f2 x = f2_fma(ru, ru, f2_mul(rv, rv));
        float x0 = fminf(fmaxf(f2_lo(x), xs_min), xs_max), x1 = fminf(fmaxf(f2_hi(x), xs_min), xs_max);
        if (!kGauss && !kMLE) {
            x0 = f2_lo(nden[i]) >= 0.f ? q.xmu : x0;
            x1 = f2_hi(nden[i]) >= 0.f ? q.xmu : x1;
        }
        xs[i] = f2_pack(x0, x1);
    }
#pragma unroll
    for (int i = 0; i < P; ++i) s[i] = f2_fma(q.beta, kGauss ? xs[i] : f2_lg2(xs[i]), q.beta_k);
    if (kGauss) {
        // log2(mu / rho) = s; log2(1 + 2^s) = max(s, 0) + log2(1 + 2^-|s|)
#pragma unroll
        for (int i = 0; i < P; ++i) {
            v[i] = s[i];
            if (!kMLE) {
                const float g0 = f2_lo(s[i]), g1 = f2_hi(s[i]);
                const f2 e = f2_pack(mufu_ex2(-fabsf(g0)), mufu_ex2(-fabsf(g1)));
                const f2 sm = log2_1p_small(e), e1 = f2_add(e, f2_both(1.f));
                v[i] = f2_add(f2_pack(fmaxf(g0, 0.f), fmaxf(g1, 0.f)),
                              f2_pack(lg2_if_large(f2_lo(sm), f2_lo(e), f2_lo(e1)), lg2_if_large(f2_hi(sm), f2_hi(e), f2_hi(e1))));
            }
        }
    } else {
        f2 r[P];
#pragma unroll
        for (int i = 0; i < P; ++i) {
            const float s0 = f2_lo(s[i]), s1 = f2_hi(s[i]);
            const f2 ep = f2_pack(mufu_ex2(s0), mufu_ex2(s1)), en = f2_pack(mufu_ex2(-s0), mufu_ex2(-s1));
            r[i] = f2_mul(f2_mul(q.Cp, xs[i]), f2_add(ep, f2_add(en, f2_both(2.f))));
        }
#pragma unroll
        for (int i = 0; i < P; ++i) {
            if (kMLE) {
                v[i] = f2_lg2(r[i]);
            } else {
                const f2 sm = log2_1p_small(r[i]), r1 = f2_add(r[i], f2_both(1.f));
                v[i] = f2_pack(lg2_if_large(f2_lo(sm), f2_lo(r[i]), f2_lo(r1)), lg2_if_large(f2_hi(sm), f2_hi(r[i]), f2_hi(r1)));
            }
        }
    }
#pragma unroll
    for (int i = 0; i < P; ++i) {
        if (kGauss || kMLE) {
            constexpr float behind = kMLE ? 0.f : 1.f;
            v[i] = f2_pack(f2_lo(nden[i]) >= 0.f ? behind : f2_lo(v[i]), f2_hi(nden[i]) >= 0.f ? behind : f2_hi(v[i]));
        }
        acc[i] = f2_fma(q.wq, v[i], acc[i]);
    }
}

// NC consecutive TMEM columns of the warp's 32 lanes.
template <int NC>
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t* r);

template <>
__device__ __forceinline__ void tmem_ld<2>(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x2.b32 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(taddr));
}

template <>
__device__ __forceinline__ void tmem_ld<4>(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr));
}

template <>
__device__ __forceinline__ void tmem_ld<8>(uint32_t taddr, uint32_t* r)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr));
}

// Bounded wait on an mbarrier phase: false (and *bad set, if given) on expiry or
// when another role of the CTA already gave up. The loop is out of line: the
// first try nearly always succeeds, and the hot loop holds only that.
constexpr long long kWaitLimit = 1ll << 26;

__device__ __noinline__ bool score_wait_loop(uint32_t bar, uint32_t parity, volatile int* bad, long long limit)
{
    for (long long i = 0; i < limit; ++i) {
        if (tc_try_wait(bar, parity)) return true;
        if ((i & 1023) == 1023 && bad && *bad) return false;
    }
    if (bad) *bad = 1;
    return false;
}

__device__ __forceinline__ bool score_wait(uint32_t bar, uint32_t parity, volatile int* bad)
{
    return tc_try_wait(bar, parity) || score_wait_loop(bar, parity, bad, kWaitLimit);
}

// The same for a converged warp, with one answer for all its lanes.
__device__ __forceinline__ bool score_wait_warp(uint32_t bar, uint32_t parity, volatile int* bad)
{
    return __all_sync(0xffffffffu, score_wait(bar, parity, bad));
}

// ---------------------------------------------------------------------------
// The scoring kernel: one persistent CTA per SM over work items (pixel chunk,
// group of 128 hypotheses), chunk-major so that the CTAs running at one time
// share the pixel tiles in L2. Warp roles:
//   warp 16, an elected lane: bulk copies of an item's hypothesis operand (40 KB, two
//     buffers) and pixel tiles (128 pixels, 24 KB, kScSlots slots);
//   warp 17, an elected lane: per tile and stage of 32 hypotheses six MMAs of M = 128
//     pixels, K = 16 (N = 96: S by US, VS, ZS; N = 32: U by XU, V by XV) into one of
//     five TMEM buffers of 96 columns U, V, a_z;
//   warps 0-15: warp w takes the 32 pixels of TMEM lane quarter w % 4 and stage
//     w / 4 of the group, kL hypotheses at a time: one pixel per lane, the
//     hypotheses packed in pairs. Four warp groups and five buffers: a group's
//     next tile is computed while it works on this one. A lane's sums over its pixels
//     are FP32 over at most kScFlush tiles, then added across lanes and from
//     there on in FP64; the four quarters' sums are added in order.
//
// What bounds it. Per SM sub-partition and 64 pairs (one warp instruction of
// packed pairs) the Fisk / MIE term costs 56 cycles of SFU time (half an rcp, one
// lg2, two ex2 per pair, one lg2 where r >= 1/8; rcp and lg2 take 8 cycles per
// warp, ex2 4) and 49 issue slots, of which the 17 packed instructions hold the
// dispatch port two cycles each; it runs in 73 cycles, the SFU 77 % busy, the
// tensor pipe 31 %. With the contractions in FP32 on the CUDA cores the term
// needed 28 packed instructions and five shared-memory loads per pixel and was
// bound by dispatch: 88 cycles. 8192 hypotheses x 465,750 pixels: 4.38 -> 3.64 ms.
// The two issuing warps run converged: with their loops inside an `if (lane == 0)` a
// stage's six MMAs, descriptors, waits and commit took longer than the arithmetic of the
// light variants, and MLE with the Gaussian residual (one rcp a pair) took 1977 us a frame
// on average there, then 1587, MIE with it 2198, then 2055 (1599 and 2128 with what
// score_pairs does for their precision); MIE / Fisk 2334, now 2306, MLE / Fisk 2190.
// Measured and not kept: the next columns' loads from tensor memory issued before the
// arithmetic on the present ones (24 more registers: MIE / Fisk 1 % faster, MLE / Fisk 1 %
// and MIE / Gaussian 5 % slower), 8 or 12 compute warps with more registers (101 and 91
// cycles against 88 with 16 at the first version), all arithmetic scalar (79
// against 73), two 64-hypothesis buffers (76), lg2(1 + r) as a polynomial on the
// FMA pipe (115 in the FP32 kernel), and a shortened register share for the two
// issuing warps (setmaxnreg; 95).
// ---------------------------------------------------------------------------
constexpr int kScWarps = 16;                              // compute warps
constexpr int kScThreads = (kScWarps + 2) * 32;
constexpr int kScSlots = 3;
constexpr int kScFlush = 64;                              // tiles summed in FP32 per lane: 64 terms, then 4 lanes
constexpr int kScHypOff = kScSlots * kScTileBytes;
constexpr int kScBarOff = kScHypOff + 2 * kScGroupBytes;
constexpr int kScRedOff = kScBarOff + 256;
constexpr int kScSmemBytes = kScRedOff + 2 * 4 * kScGroupHyps * 8;
constexpr int kScStageCols = 3 * kScStageHyps;            // TMEM columns of a buffer
constexpr int kScBufs = 5;
constexpr int kScTmemCols = 512;                          // the buffers' 480, rounded up to a power of two

struct ScItem {
    int t0, cnt, hyps;                                    // first tile, tiles, hypotheses
};

template <int kL, bool kMLE, bool kGauss>
__global__ void __launch_bounds__(kScThreads, 1) k_score(DevParams p, DevState s, int log_idx)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    const uint32_t sb = smem_addr(smem), ring = sb, hyp_s = sb + kScHypOff, bars = sb + kScBarOff;
    const uint32_t full = bars, empty = full + 8 * kScSlots, hfull = empty + 8 * kScSlots, hempty = hfull + 16;
    const uint32_t afull = hempty + 16, aempty = afull + 8 * kScBufs, done = aempty + 8 * kScBufs;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kScBarOff + 200);
    volatile int& bad = *reinterpret_cast<volatile int*>(smem + kScBarOff + 204);
    volatile int& last = *reinterpret_cast<volatile int*>(smem + kScBarOff + 208);
    double* red = reinterpret_cast<double*>(smem + kScRedOff);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n_hyp = *s.n_hyp, n_pix = *s.pix_count;
    if (log_idx >= 0 && blockIdx.x == 0 && threadIdx.x == 0) {
        s.score_log[2 * log_idx] = n_hyp;
        s.score_log[2 * log_idx + 1] = n_pix;
    }
    const int n_tiles = (n_pix + kScTilePix - 1) / kScTilePix;
    const int few = *s.few_chunks, n_groups = (n_hyp + kScGroupHyps - 1) / kScGroupHyps, n_chunks = few ? few : s.n_chunks;
    const int n_items = n_groups * n_chunks;
    if (blockIdx.x >= n_items) return;
    auto item = [&](int u) {
        const int chunk = u / n_groups, group = u % n_groups;
        ScItem w;
        w.t0 = (int)((long long)n_tiles * chunk / n_chunks);
        w.cnt = (int)((long long)n_tiles * (chunk + 1) / n_chunks) - w.t0;
        w.hyps = min(kScGroupHyps, n_hyp - group * kScGroupHyps);
        return w;
    };
    if (threadIdx.x == 0) {
        for (int i = 0; i < kScSlots; ++i) {
            tc_mbar_init(full + 8 * i, 1);
            tc_mbar_init(empty + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc_mbar_init(hfull + 8 * i, 1);
            tc_mbar_init(hempty + 8 * i, 1);
        }
        for (int i = 0; i < kScBufs; ++i) {
            tc_mbar_init(afull + 8 * i, 1);
            tc_mbar_init(aempty + 8 * i, kScWarps / kScGroupStages);
        }
        tc_mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        bad = 0;
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                     "r"((uint32_t)kScTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == kScWarps) {
        // loader: n counts tiles, w work items (those with pixels)
        uint32_t n = 0, w = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < n_items && ok; u += gridDim.x) {
            const ScItem it = item(u);
            if (it.cnt == 0) continue;
            const uint32_t hb = w & 1, bytes = (it.hyps + kScStageHyps - 1) / kScStageHyps * kScStageBytes;
            if (w >= 2) ok = score_wait_warp(hempty + 8 * hb, ((w >> 1) - 1) & 1, &bad);
            if (!ok) break;
            tc_expect_tx_elect(hfull + 8 * hb, bytes);
            tc_bulk_g2s_elect(hyp_s + hb * kScGroupBytes, s.sc_hyp + (size_t)(u % n_groups) * kScGroupBytes, bytes, hfull + 8 * hb);
            ++w;
            for (int k = 0; k < it.cnt; ++k, ++n) {
                const uint32_t slot = n % kScSlots;
                if (n >= kScSlots) ok = score_wait_warp(empty + 8 * slot, ((n / kScSlots) - 1) & 1, &bad);
                if (!ok) break;
                tc_expect_tx_elect(full + 8 * slot, kScTileBytes);
                tc_bulk_g2s_elect(ring + slot * kScTileBytes, s.sc_pix + (size_t)(it.t0 + k) * kScTileBytes, kScTileBytes, full + 8 * slot);
            }
        }
        // the last copies may still be landing when another role gave up
        for (uint32_t j = n > kScSlots ? n - kScSlots : 0; j < n; ++j)
            score_wait(full + 8 * (j % kScSlots), (j / kScSlots) & 1, nullptr);
        for (uint32_t j = w > 2 ? w - 2 : 0; j < w; ++j) score_wait(hfull + 8 * (j & 1), (j >> 1) & 1, nullptr);
    } else if (warp == kScWarps + 1) {
        // MMA issuer: stages in TMEM buffers 0 .. kScBufs - 1 in turn, tb the next one's
        constexpr uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kScTilePix >> 4) << 24);
        constexpr uint32_t idS = id | ((uint32_t)(3 * kScStageHyps >> 3) << 17), idX = id | ((uint32_t)(kScStageHyps >> 3) << 17);
        constexpr uint32_t kA = kScTilePix * 16;                       // bytes of a column block of A
        uint32_t n = 0, w = 0, m = 0;
        bool ok = true;
        for (int u = blockIdx.x; u < n_items && ok; u += gridDim.x) {
            const ScItem it = item(u);
            if (it.cnt == 0) continue;
            const uint32_t hb = w & 1;
            ok = score_wait_warp(hfull + 8 * hb, (w >> 1) & 1, &bad);
            const int stages = (it.hyps + kScStageHyps - 1) / kScStageHyps;
            for (int k = 0; k < it.cnt && ok; ++k, ++n) {
                const uint32_t slot = n % kScSlots, a = ring + slot * kScTileBytes;
                ok = score_wait_warp(full + 8 * slot, (n / kScSlots) & 1, &bad);
                for (int st = 0; st < stages && ok; ++st, ++m) {
                    const uint32_t tb = m % kScBufs;
                    if (m >= kScBufs) ok = score_wait_warp(aempty + 8 * tb, ((m / kScBufs) - 1) & 1, &bad);
                    if (!ok) break;
                    tc_fence_after();
                    const uint32_t b = hyp_s + hb * kScGroupBytes + st * kScStageBytes, d = tmem + tb * kScStageCols;
                    // column blocks of A: S at 0, U at 4, V at 8; each block's small products are in its
                    // first two column blocks, the large ones of U and V in the last two of U and V
                    auto mma_s = [&](int half, uint32_t acc) {
                        tc_mma_elect(d, tc_desc(a + 2 * half * kA, kA, 128), tc_desc(b + 2 * half * kScHypSBlock, kScHypSBlock, 128), idS, acc);
                    };
                    auto mma_x = [&](int v, int half) {
                        tc_mma_elect(d + v * kScStageHyps, tc_desc(a + (4 + 4 * v + 2 * half) * kA, kA, 128),
                                     tc_desc(b + (v ? kScHypVOff : kScHypUOff) + 2 * half * kScHypXBlock, kScHypXBlock, 128), idX, 1u);
                    };
                    mma_s(0, 0u);
                    mma_s(1, 1u);
                    mma_x(0, 0);
                    mma_x(1, 0);
                    mma_x(0, 1);
                    mma_x(1, 1);
                    tc_commit_elect(afull + 8 * tb);
                }
                if (ok) tc_commit_elect(empty + 8 * slot);
            }
            if (ok) tc_commit_elect(hempty + 8 * hb);
            ++w;
        }
        tc_commit_elect(done);                // arrives once every MMA issued above has completed
        score_wait(done, 0, nullptr);
    } else {
        const int quarter = warp & 3, wg = warp >> 2;
        const uint32_t tlane = tmem + ((uint32_t)(quarter * 32) << 16);
        const float xs_min = p.xs_min, xs_max = p.xs_max;
        const bool wild = *s.sc_wild != 0;
        uint32_t tb = 0, phase = 0;                          // TMEM buffer of the next tile's stage 0 and its phase
        int buf = 0;
        bool go = true;
        f2 acc[kScStageHyps / 2];
        // tiles [t0, t1) of `stages` stages: the lane's pixel of each against the warp's 32 hypotheses
        auto tiles = [&](auto is_wild, int t0, int t1, int stages) {
            constexpr bool kWild = decltype(is_wild)::value;
            int j = t0 * kScTilePix + quarter * 32 + lane;
            // a lane past the last pixel: weight 0 and a finite term, whatever its operand row holds
            float4 cst;
            float xmu;
            auto load_const = [&]() {
                const bool in = j < n_pix;
                cst = in ? __ldg(s.sc_cst + j) : make_float4(0.f, 0.f, 1.f, 0.f);
                xmu = in ? __ldg(s.sc_xmu + j) : 1.f;
            };
            load_const();
            for (int t = t0; t < t1; ++t) {
                const PixConst q{f2_both(cst.x), f2_both(cst.y), f2_both(cst.z), f2_both(cst.w), xmu};
                j += kScTilePix;
                load_const();
                // every lane polls; the warp proceeds only together (tcgen05.ld is warp-wide)
                const uint32_t b = tb + wg, bw = b >= kScBufs, buf8 = 8 * (b - bw * kScBufs);
                go = __all_sync(0xffffffffu, score_wait(afull + buf8, phase ^ bw, &bad));
                if (!go) return;
                tc_fence_after();
                const uint32_t cols = tlane + buf8 * (kScStageCols / 8);
                tb += stages;
                if (tb >= kScBufs) {
                    tb -= kScBufs;
                    phase ^= 1u;
                }
#pragma unroll
                for (int part = 0; part < kScStageHyps / kL; ++part) {
                    uint32_t U[kL], V[kL], Z[kL];
                    tmem_ld<kL>(cols + part * kL, U);
                    tmem_ld<kL>(cols + part * kL + kScStageHyps, V);
                    tmem_ld<kL>(cols + part * kL + 2 * kScStageHyps, Z);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    tc_hold<kL>(U);
                    tc_hold<kL>(V);
                    tc_hold<kL>(Z);
                    if (part == kScStageHyps / kL - 1) {      // the warp's columns are in registers
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) tc_arrive(aempty + buf8);
                    }
                    score_pairs<kL / 2, kMLE, kGauss, kWild>(U, V, Z, q, xs_min, xs_max, &acc[part * (kL / 2)]);
                }
            }
        };
        // every warp passes every item's barrier, also after a wait gave up (go stays false)
        for (int u = blockIdx.x; u < n_items; u += gridDim.x) {
            const ScItem it = item(u);
            double tot = 0.0;
            const int stages = (it.hyps + kScStageHyps - 1) / kScStageHyps;
            if (wg >= stages) {                              // nothing of this group for the warp: keep count of the buffers
                const uint32_t b = tb + (uint32_t)(it.cnt * stages);
                phase ^= (b / kScBufs) & 1u;
                tb = b % kScBufs;
            }
            for (int k0 = 0; k0 < it.cnt && wg < stages && go; k0 += kScFlush) {
                const int k1 = min(k0 + kScFlush, it.cnt);
#pragma unroll
                for (int i = 0; i < kScStageHyps / 2; ++i) acc[i] = 0ull;
                if (wild) tiles(std::true_type{}, it.t0 + k0, it.t0 + k1, stages);
                else tiles(std::false_type{}, it.t0 + k0, it.t0 + k1, stages);
                // sums over the warp's 32 lanes: at each step a lane keeps half of its values and
                // adds the partner's, so lane l ends with the sum of value l (FP32 over 4 lanes, then FP64)
                float f[32];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    f[2 * i] = f2_lo(acc[i]);
                    f[2 * i + 1] = f2_hi(acc[i]);
                }
#pragma unroll
                for (int o = 16, m = 16; o >= 8; o >>= 1, m >>= 1)
#pragma unroll
                    for (int i = 0; i < m; ++i) {
                        const bool up = (lane & o) != 0;
                        const float send = up ? f[i] : f[i + m], keep = up ? f[i + m] : f[i];
                        f[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                double d[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) d[i] = (double)f[i];
#pragma unroll
                for (int o = 4, m = 4; o >= 1; o >>= 1, m >>= 1)
#pragma unroll
                    for (int i = 0; i < m; ++i) {
                        const bool up = (lane & o) != 0;
                        const double send = up ? d[i] : d[i + m], keep = up ? d[i + m] : d[i];
                        d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                    }
                tot += d[0];
            }
            red[(buf * 4 + quarter) * kScGroupHyps + wg * kScStageHyps + lane] = tot;
            asm volatile("bar.sync 1, %0;" ::"n"(kScWarps * 32) : "memory");
            if (warp < kScGroupHyps / 32) {
                const int h = threadIdx.x, chunk = u / n_groups, group = u % n_groups;
                double* part = s.partial + group * kScGroupHyps + h;
                if (h < it.hyps) {
                    const double* r = red + buf * 4 * kScGroupHyps + h;
                    const double v = ((r[0] + r[kScGroupHyps]) + r[2 * kScGroupHyps]) + r[3 * kScGroupHyps];
                    part[(size_t)chunk * p.S] = -v * 0.69314718055994531;
                }
                // the CTA that finishes a group's last chunk adds the chunks in order (no CTA waits)
                __threadfence();
                asm volatile("bar.sync 2, %0;" ::"n"(kScGroupHyps) : "memory");
                if (h == 0) last = atomicAdd(s.score_done + group, 1) == n_chunks - 1;
                asm volatile("bar.sync 2, %0;" ::"n"(kScGroupHyps) : "memory");
                if (last) {
                    __threadfence();
                    if (h == 0) s.score_done[group] = 0;
                    if (h < it.hyps) {
                        double v = 0.0;
                        for (int c = 0; c < n_chunks; c += 8) {
                            double a[8];
#pragma unroll
                            for (int i = 0; i < 8; ++i) a[i] = c + i < n_chunks ? __ldcg(part + (size_t)(c + i) * p.S) : 0.0;
#pragma unroll
                            for (int i = 0; i < 8; ++i) v += a[i];
                        }
                        s.scores[group * kScGroupHyps + h] = v;
                    }
                }
            }
            buf ^= 1;          // the next item's sums go to the other buffer, so one barrier per item suffices
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)kScTmemCols));
    }
    if (threadIdx.x == 0 && bad) atomicOr(s.status + 3, kStatusTimeout);
}

static int g_num_sms = 0;

static int num_sms()
{
    if (g_num_sms == 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || g_num_sms <= 0)
            g_num_sms = 152;
    }
    return g_num_sms;
}

// Pixel chunks of at most `waves` work items (pixel chunk x group of 128
// hypotheses) per SM: the count with the shortest schedule, rounds of items times
// an item's tiles plus kItemTiles, the cost of starting and flushing an item in
// tiles. Few items leave the last round partly empty, many pay that cost each time.
int score_chunks_for(int S, int N, int waves)
{
    constexpr double kItemTiles = 1.5;
    const int groups = (S + kScGroupHyps - 1) / kScGroupHyps, tiles = (N + kScTilePix - 1) / kScTilePix, sms = num_sms();
    const int most = std::max(1, std::min(sms * waves / groups, tiles));
    int best = most;
    double best_cost = 1e300;
    for (int c = 1; c <= most; ++c) {
        const double cost = ((groups * (long long)c + sms - 1) / sms) * ((tiles + c - 1) / c + kItemTiles);
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

int score_ctas() { return num_sms(); }

int score_chunks(int S, int N) { return score_chunks_for(S, N, kScoreDefaultWaves); }

// Largest chunk count a window accepts (and its partial sums are sized for).
int score_chunks_max(int S, int N)
{
    const int groups = (S + kScGroupHyps - 1) / kScGroupHyps, px = (N + kScTilePix - 1) / kScTilePix;
    int most = std::max(1, std::min(num_sms() * kTuneMaxWaves / groups, px));
    for (int hpt = 2; hpt <= 8; hpt *= 2) {
        const int tiles = (S + 256 * hpt - 1) / (256 * hpt), blocks = hpt == 8 ? 1 : (hpt == 4 ? 2 : 3);
        most = std::max(most, std::min((num_sms() * blocks * kTuneMaxWaves + tiles - 1) / tiles, N));
    }
    return most;
}

template <int kL, bool kMLE, bool kGauss>
static void launch_score_as(const DevParams& p, const DevState& s, int li, cudaStream_t st)
{
    // the dynamic shared-memory limit is raised once per device
    constexpr int kMaxDevices = 64;
    static std::mutex mutex;
    static bool raised[kMaxDevices];
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kMaxDevices) {
        std::lock_guard<std::mutex> lock(mutex);
        if (!raised[dev])
            raised[dev] = cudaFuncSetAttribute(k_score<kL, kMLE, kGauss>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kScSmemBytes) == cudaSuccess;
    }
    // a frame with fewer groups may have more items than a full one
    const int groups = (p.S + kScGroupHyps - 1) / kScGroupHyps, tiles = (p.N + kScTilePix - 1) / kScTilePix;
    const long long items = std::max((long long)groups * s.n_chunks, (long long)(groups - 1) * std::min(s.chunks_max, tiles));
    k_score<kL, kMLE, kGauss><<<(unsigned)std::min<long long>(items, num_sms()), kScThreads, kScSmemBytes, st>>>(p, s, li);
}

template <int kL>
static void launch_score_shape(const DevParams& p, const DevState& s, int li, cudaStream_t st)
{
    const bool mle = p.criterion == VOLDOR_CRITERION_MLE, gauss = p.residual == VOLDOR_RESIDUAL_GAUSSIAN;
    if (gauss && mle) launch_score_as<kL, true, true>(p, s, li, st);
    else if (gauss) launch_score_as<kL, false, true>(p, s, li, st);
    else if (mle) launch_score_as<kL, true, false>(p, s, li, st);
    else launch_score_as<kL, false, false>(p, s, li, st);
}

void launch_score(const DevParams& p, const DevState& s, int log_idx, cudaStream_t st)
{
    const int li = log_idx < kScoreLogMax ? log_idx : -1;
    if (s.score_hpt == 4) launch_score_shape<4>(p, s, li, st);
    else if (s.score_hpt == 2) launch_score_shape<2>(p, s, li, st);
    else launch_score_shape<8>(p, s, li, st);
}


// ---------------------------------------------------------------------------
// Allocation-free dense scoring.
//
// Some callers cannot allocate device memory at the time they want a score:
// code running inside a CUDA stream capture that must not add allocation
// nodes, a host that hands the GPU to this library under a fixed memory
// budget, or a caller whose own allocator owns all device memory. For them,
// voldor_score_records_noalloc scores caller-given pixel records against
// caller-given hypotheses by the same formula, in plain FP32 (no tensor cores, a
// reciprocal to each pair): its scores and k_score's agree within the bound on dense
// scores, not bit for bit. It takes its only scratch (the per-chunk partial sums) from the file-scope
// array below, which every GPU that loads this library holds until the
// process exits.
// ---------------------------------------------------------------------------
constexpr int kStaticMaxHyps = 8192;
constexpr int kStaticChunks = 64;
static __device__ __align__(256) double g_static_partials[kStaticChunks * kStaticMaxHyps];   // 4 MiB

__global__ void __launch_bounds__(kScoreThreads, kScoreBlocksPerSM)
k_score_records(const float4* __restrict__ pix, int n_pix, const float* __restrict__ hyps, int n_hyp, float xs_min,
                float xs_max, double* __restrict__ partial)
{
    const int tile0 = blockIdx.x * kScoreHypsPerBlock;
    if (tile0 >= n_hyp) return;
    const int chunk = blockIdx.y, n_chunks = gridDim.y;
    const long long lo = (long long)n_pix * chunk / n_chunks;
    const long long hi = (long long)n_pix * (chunk + 1) / n_chunks;
    HypF hy[kScoreHypsPerThread];
#pragma unroll
    for (int i = 0; i < kScoreHypsPerThread; ++i) {
        const float* f = hyps + (size_t)min(tile0 + i * kScoreThreads + (int)threadIdx.x, n_hyp - 1) * 12;
        hy[i] = HypF{f[0], f[1], f[2], f[3], f[4], f[5], f[6], f[7], f[8], f[9], f[10], f[11]};
    }
    double acc[kScoreHypsPerThread];
    float facc[kScoreHypsPerThread];
#pragma unroll
    for (int i = 0; i < kScoreHypsPerThread; ++i) { acc[i] = 0.0; facc[i] = 0.f; }
    long long j = lo;
    while (j < hi) {
        const long long jend = min(hi, j + 32);
        for (; j < jend; ++j) {
            const float4 a = __ldg(pix + 3 * j);
            const float4 b = __ldg(pix + 3 * j + 1);
            const float wq = __ldg(reinterpret_cast<const float*>(pix + 3 * j + 2));
#pragma unroll
            for (int i = 0; i < kScoreHypsPerThread; ++i)
                facc[i] = fmaf(wq, pair_term2(hy[i], a, b, xs_min, xs_max), facc[i]);
        }
#pragma unroll
        for (int i = 0; i < kScoreHypsPerThread; ++i) { acc[i] += (double)facc[i]; facc[i] = 0.f; }
    }
#pragma unroll
    for (int i = 0; i < kScoreHypsPerThread; ++i) {
        const int h = tile0 + i * kScoreThreads + threadIdx.x;
        if (h < n_hyp) partial[(size_t)chunk * kStaticMaxHyps + h] = -acc[i] * 0.69314718055994531;
    }
}

__global__ void k_reduce_records(const double* __restrict__ partial, int n_hyp, int n_chunks, double* __restrict__ L)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= n_hyp) return;
    double v = 0.0;
    for (int c = 0; c < n_chunks; ++c) v += partial[(size_t)c * kStaticMaxHyps + h];
    L[h] = v;
}

// Device address of g_static_partials, looked up once per device with that
// device current (a host-side reference to the array is only a stand-in).
constexpr int kStaticMaxDevices = 64;
static double* g_static_ptr[kStaticMaxDevices];
static std::mutex g_static_mutex;

static cudaError_t static_partials(double** out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kStaticMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_static_partials);
        if (e != cudaSuccess) return e;
        g_static_ptr[dev] = static_cast<double*>(p);
    }
    *out = g_static_ptr[dev];
    return cudaSuccess;
}

}  // namespace vd

extern "C" voldor_status voldor_score_records_noalloc(const float* records, int n_pix, const float* hyps, int n_hyps,
                                                      double xs_min, double xs_max, double* L, void* cuda_stream)
{
    using namespace vd;
    if (!records || !hyps || !L || n_pix < 0 || n_hyps < 1) return VOLDOR_ERR_INVALID_ARG;
    if (n_hyps > kStaticMaxHyps) return VOLDOR_ERR_INVALID_ARG;
    // the kernel reads records as float4 and writes L as double
    if (((uintptr_t)records & 15u) || ((uintptr_t)hyps & 3u) || ((uintptr_t)L & 7u)) return VOLDOR_ERR_INVALID_ARG;
    if (!(xs_min > 0.0) || !(xs_max > xs_min) || !std::isfinite(xs_max)) return VOLDOR_ERR_INVALID_ARG;
    double* partial = nullptr;
    if (static_partials(&partial) != cudaSuccess) {
        cudaGetLastError();
        return VOLDOR_ERR_CUDA;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const int tiles = (n_hyps + kScoreHypsPerBlock - 1) / kScoreHypsPerBlock;
    k_score_records<<<dim3(tiles, kStaticChunks), kScoreThreads, 0, st>>>(
        reinterpret_cast<const float4*>(records), n_pix, hyps, n_hyps, (float)xs_min, (float)xs_max, partial);
    k_reduce_records<<<(n_hyps + 255) / 256, 256, 0, st>>>(partial, n_hyps, kStaticChunks, L);
    if (cudaGetLastError() != cudaSuccess) return VOLDOR_ERR_CUDA;
    return VOLDOR_OK;
}

// ---------------------------------------------------------------------------
// Diagnostic: SFU (MUFU) throughput of this GPU in results per SM clock, for
// the roofline of the dense scoring. One wave of blocks (4 per SM, 256
// threads) runs 16 independent chains of one SFU op per thread; the whole
// grid is timed with CUDA events, and the SM clock during the run is measured
// in the kernel (clock64 cycles over globaltimer nanoseconds of each block,
// median over blocks), so results per SM clock = results / (grid time x SM
// clock x SMs) holds at whatever clock the GPU ran.
// ---------------------------------------------------------------------------
namespace vd {
constexpr int kProbeChains = 16;

// One SFU op per chain step, fixed at compile time: with the op chosen at run
// time inside the loop the compiler predicates the branches and issues every
// branch's SFU instruction on each step.
template <int OP>
__device__ __forceinline__ float sfu_step(float v)
{
    float y;
    if constexpr (OP == 0) {          // exp2(-|v|): stays in [0.5, 1)
        asm volatile("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-fabsf(v)));
    } else if constexpr (OP == 1) {   // log2(v) + 1.5: converges to ~3.2, stays normal
        asm volatile("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(v));
        y += 1.5f;
    } else {                          // 1 / (-v): alternates between two normal values
        asm volatile("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(-v));
    }
    return y;
}

__device__ __forceinline__ unsigned long long global_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

template <int OP>
__global__ void __launch_bounds__(256) k_sfu_probe(int iters, float seed, float* sink, long long* clk)
{
    float v[kProbeChains];
#pragma unroll
    for (int i = 0; i < kProbeChains; ++i) v[i] = seed + 0.001f * (float)((threadIdx.x + i) & 63);
    __syncthreads();
    const long long c0 = clock64();
    const unsigned long long g0 = global_ns();
    for (int it = 0; it < iters; ++it) {
#pragma unroll
        for (int i = 0; i < kProbeChains; ++i) v[i] = sfu_step<OP>(v[i]);
    }
    __syncthreads();
    const long long c1 = clock64();
    const unsigned long long g1 = global_ns();
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kProbeChains; ++i) acc += v[i];
    if (acc == 1234.5f) sink[threadIdx.x] = acc;     // keeps the chains alive
    if (threadIdx.x == 0) {
        clk[2 * blockIdx.x] = c1 - c0;
        clk[2 * blockIdx.x + 1] = (long long)(g1 - g0);
    }
}

void launch_sfu_probe(int op, int blocks, int threads, int iters, float seed, float* sink, long long* clk)
{
    if (op == 0) k_sfu_probe<0><<<blocks, threads>>>(iters, seed, sink, clk);
    else if (op == 1) k_sfu_probe<1><<<blocks, threads>>>(iters, seed, sink, clk);
    else k_sfu_probe<2><<<blocks, threads>>>(iters, seed, sink, clk);
}
}  // namespace vd

extern "C" voldor_status voldor_probe_sfu_rate(int op, double* results_per_sm_clock, double* sm_mhz)
{
    using namespace vd;
    if (!results_per_sm_clock || op < 0 || op > 2) return VOLDOR_ERR_INVALID_ARG;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return VOLDOR_ERR_CUDA;
    const int blocks = sms * 4, threads = 256, iters = 4096;
    float* sink = nullptr;
    long long* clk = nullptr;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (cudaMalloc(&sink, threads * sizeof(float)) != cudaSuccess) return VOLDOR_ERR_OOM;
    if (cudaMalloc(&clk, 2 * blocks * sizeof(long long)) != cudaSuccess) { cudaFree(sink); return VOLDOR_ERR_OOM; }
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    const float seed = op == 1 ? 1.5f : 0.75f;
    float ms = 0.f;
    std::vector<long long> h(2 * blocks);
    if (e == cudaSuccess) {
        launch_sfu_probe(op, blocks, threads, 256, seed, sink, clk);          // warm-up
        cudaEventRecord(e0);
        launch_sfu_probe(op, blocks, threads, iters, seed, sink, clk);
        cudaEventRecord(e1);
        e = cudaEventSynchronize(e1);
    }
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
    if (e == cudaSuccess) e = cudaMemcpy(h.data(), clk, h.size() * sizeof(long long), cudaMemcpyDeviceToHost);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    cudaFree(sink);
    cudaFree(clk);
    if (e != cudaSuccess || !(ms > 0.f)) return VOLDOR_ERR_CUDA;
    std::vector<double> mhz;
    for (int b = 0; b < blocks; ++b)
        if (h[2 * b + 1] > 0) mhz.push_back(1e3 * (double)h[2 * b] / (double)h[2 * b + 1]);
    if (mhz.empty()) return VOLDOR_ERR_INTERNAL;
    std::nth_element(mhz.begin(), mhz.begin() + mhz.size() / 2, mhz.end());
    const double f = mhz[mhz.size() / 2];                      // MHz
    const double results = (double)blocks * threads * (double)kProbeChains * iters;
    *results_per_sm_clock = results / ((double)ms * 1e-3 * f * 1e6 * sms);
    if (sm_mhz) *sm_mhz = f;
    return VOLDOR_OK;
}

// ---------------------------------------------------------------------------
// Diagnostic: the expiry path of the bounded mbarrier waits.
// ---------------------------------------------------------------------------
namespace vd {
// Bounded-wait probe: every thread of one block waits, with the scoring
// kernel's bounded wait, on the first phase of an mbarrier that nothing
// arrives on, for `polls` polls; out[0] = number of threads that gave up,
// out[1] = SM cycles the wait took on thread 0.
__global__ void k_wait_probe(long long polls, long long* out)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        tc_mbar_init(smem_addr(&bar), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const long long t0 = clock64();
    const bool done = score_wait_loop(smem_addr(&bar), 0, nullptr, polls);
    const long long t1 = clock64();
    const int gave_up = __syncthreads_count(!done);
    if (threadIdx.x == 0) {
        out[0] = gave_up;
        out[1] = t1 - t0;
    }
}

}  // namespace vd

extern "C" voldor_status voldor_probe_bounded_wait(long long polls, long long* cycles)
{
    using namespace vd;
    if (polls < 0 || polls > kWaitLimit) return VOLDOR_ERR_INVALID_ARG;
    long long* d = nullptr;
    if (cudaMalloc(&d, 2 * sizeof(long long)) != cudaSuccess) return VOLDOR_ERR_OOM;
    k_wait_probe<<<1, 128>>>(polls, d);
    long long h[2] = {0, 0};
    const cudaError_t e = cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost);
    cudaFree(d);
    if (e != cudaSuccess || cudaGetLastError() != cudaSuccess) return VOLDOR_ERR_CUDA;
    if (cycles) *cycles = h[1];
    return h[0] == 128 ? VOLDOR_ERR_TIMEOUT : (h[0] == 0 ? VOLDOR_OK : VOLDOR_ERR_INTERNAL);
}

