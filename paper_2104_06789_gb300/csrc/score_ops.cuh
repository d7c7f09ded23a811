// Operands of the dense scoring's tensor-core projection.
//
// For a pixel with normalised coordinates p = (x, y, 1) (y scaled by fy/fx),
// inverse depth w and observed flow (ut, vt) (all over fx, camera t-1) and a
// hypothesis E = R - I, t (scaled alike), the scoring needs
//   a_z = E_z p + t_z w,   U = X a_z - a_x + ut,   V = Y a_z - a_y + vt
// with X = x + ut, Y = y + vt: U / (1 + a_z) and V / (1 + a_z) are the residual
// over fx. All three are linear in the hypothesis once the products X x, X y,
// X w (and Y's) count as pixel features. Around a reference pose (E0, t0), the frame's
// current one or the identity, with d = (E, t) - (E0, t0):
//   a_z = a_z0 + (d_z . (x, y, w, 1))
//   U   = U0   + d_z . (X x, X y, X w, X) - d_x . (x, y, w, 1)
// so the large terms that cancel in U are formed once per pixel in float-float
// (a_z0, U0, V0), and the hypotheses that matter multiply small differences.
//
// BF16 holds 8 significant bits, so every feature f and coefficient c is cut
// into three slices f = fh + fm + fl (a float-float value to 2^-26, an FP32
// value exactly), and f c becomes the six products of at least 2^-24 weight
// (hl, lh, mm | hm, mh | hh). The tensor core adds the 16 products of an MMA step
// to the FP32 accumulator and truncates, so the order matters: the small products
// come first, and all the large ones (hh) of a value share its last step, where
// they cancel before the one truncation that counts.
//
// Pixel operand (A), one row of 96 columns: block S of features (x, y, w, 1,
// a_z0), block U of (X x, X y, X w, X, U0) and once more the large slices of (x, y,
// w, 1), block V of (Y x, Y y, Y w, Y, V0) and the same.
// Hypothesis operand (B): blocks US, VS, ZS (coefficients of U, V, a_z) pair with
// S, blocks XU and XV with U and V. The large coefficients of x, y, w, 1 in U and V
// are in XU and XV, not in US and VS. Both operands lie in 8 x 8 core matrices,
// K-major: [column block of 8][row / 8][row % 8][8]; a stage of 32 hypotheses
// holds US, VS and ZS as 96 rows of one operand, so that one MMA of N = 96
// multiplies S by all three, then XU and XV as 32 rows each.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "df32.cuh"

namespace vd {

constexpr int kScTilePix = 128;                          // pixels of a tile (MMA M)
constexpr int kScPixCols = 96;
constexpr int kScTileBytes = kScTilePix * kScPixCols * 2;          // 24 KB
constexpr int kScStageHyps = 32;                         // hypotheses of a TMEM stage
constexpr int kScHypSBlock = 3 * kScStageHyps * 16;      // bytes of a column block of US, VS, ZS
constexpr int kScHypXBlock = kScStageHyps * 16;          // of XU or XV
constexpr int kScHypUOff = 4 * kScHypSBlock, kScHypVOff = kScHypUOff + 4 * kScHypXBlock;
constexpr int kScStageBytes = kScHypVOff + 4 * kScHypXBlock;       // 10 KB
constexpr int kScGroupStages = 4;
constexpr int kScGroupHyps = kScGroupStages * kScStageHyps;        // hypotheses of a work item
constexpr int kScGroupBytes = kScGroupStages * kScStageBytes;

struct Slice3 {
    __nv_bfloat16 h, m, l;
};

// hi + lo = h + m + l to about 2^-26 (exactly for lo = 0 within BF16's range)
__device__ __forceinline__ Slice3 slice3(float hi, float lo)
{
    Slice3 s;
    s.h = __float2bfloat16_rn(hi);
    float r = __fadd_rn(__fsub_rn(hi, __bfloat162float(s.h)), lo);
    s.m = __float2bfloat16_rn(r);
    r = __fsub_rn(r, __bfloat162float(s.m));
    s.l = __float2bfloat16_rn(r);
    return s;
}

__device__ __forceinline__ Slice3 slice3(DF v) { return slice3(v.hi, v.lo); }

// Block S of a pixel: the 32 columns of (x, y, w), the constant 1 (whose
// coefficient is sliced) and the reference a_z0 (whose coefficient is 1).
__device__ __forceinline__ void pixel_block_s(const Slice3* f, const Slice3& ref, __nv_bfloat16* o)
{
    const __nv_bfloat16 one = __float2bfloat16_rn(1.f), zero = __float2bfloat16_rn(0.f);
    int k = 0;
#pragma unroll
    for (; k < 8; ++k) o[k] = zero;
#pragma unroll
    for (int i = 0; i < 3; ++i) { o[k++] = f[i].h; o[k++] = f[i].l; o[k++] = f[i].m; }
    o[k++] = one;
    o[k++] = ref.l;
#pragma unroll
    for (int i = 0; i < 3; ++i) { o[k++] = f[i].h; o[k++] = f[i].m; }
    o[k++] = one;
    o[k++] = ref.m;
#pragma unroll
    for (int i = 0; i < 3; ++i) o[k++] = f[i].h;
    o[k++] = one;
    o[k++] = ref.h;
}

// Coefficients of block S: c of (x, y, w), c1 of 1, and 1 or 0 of a_z0; a_z's row has
// the large ones too (else 0: they are in XU / XV).
__device__ __forceinline__ void hyp_block_s(const Slice3* c, const Slice3& c1, bool az, __nv_bfloat16* o)
{
    const __nv_bfloat16 r = __float2bfloat16_rn(az ? 1.f : 0.f), zero = __float2bfloat16_rn(0.f);
    int k = 0;
#pragma unroll
    for (; k < 8; ++k) o[k] = zero;
#pragma unroll
    for (int i = 0; i < 3; ++i) { o[k++] = c[i].l; o[k++] = c[i].h; o[k++] = c[i].m; }
    o[k++] = c1.l;
    o[k++] = r;
#pragma unroll
    for (int i = 0; i < 3; ++i) { o[k++] = c[i].m; o[k++] = c[i].h; }
    o[k++] = c1.m;
    o[k++] = r;
#pragma unroll
    for (int i = 0; i < 3; ++i) o[k++] = az ? c[i].h : zero;
    o[k++] = az ? c1.h : zero;
    o[k++] = r;
}

// Block U (or V) of a pixel: f = (X x, X y, X w, X), the reference U0, and the large
// slices of s = (x, y, w) and 1.
__device__ __forceinline__ void pixel_block_x(const Slice3* f, const Slice3& ref, const Slice3* s, __nv_bfloat16* o)
{
    int k = 0;
    o[k++] = __float2bfloat16_rn(0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) { o[k++] = f[i].h; o[k++] = f[i].l; o[k++] = f[i].m; }
    o[k++] = ref.l;
#pragma unroll
    for (int i = 0; i < 4; ++i) { o[k++] = f[i].h; o[k++] = f[i].m; }
    o[k++] = ref.m;
#pragma unroll
    for (int i = 0; i < 4; ++i) o[k++] = f[i].h;
    o[k++] = ref.h;
#pragma unroll
    for (int i = 0; i < 3; ++i) o[k++] = s[i].h;
    o[k++] = __float2bfloat16_rn(1.f);
}

// Its coefficients: z of f, and the large ones of a = (x, y, w), a1 of 1.
__device__ __forceinline__ void hyp_block_x(const Slice3* z, const Slice3* a, const Slice3& a1, __nv_bfloat16* o)
{
    const __nv_bfloat16 one = __float2bfloat16_rn(1.f);
    int k = 0;
    o[k++] = __float2bfloat16_rn(0.f);
#pragma unroll
    for (int i = 0; i < 4; ++i) { o[k++] = z[i].l; o[k++] = z[i].h; o[k++] = z[i].m; }
    o[k++] = one;
#pragma unroll
    for (int i = 0; i < 4; ++i) { o[k++] = z[i].m; o[k++] = z[i].h; }
    o[k++] = one;
#pragma unroll
    for (int i = 0; i < 4; ++i) o[k++] = z[i].h;
    o[k++] = one;
#pragma unroll
    for (int i = 0; i < 3; ++i) o[k++] = a[i].h;
    o[k++] = a1.h;
}

// The one truncation to 24 bits lowers |U|, |V| and |a_z| by half a unit in the last
// place on average, a relative 2^-24 / (2 ln 2) = 4.3e-8 for mantissas spread evenly
// over their logarithm. The coefficients and the references carry that much more, which
// leaves the scores without the bias: measured against 64 bits, the mean relative error
// of the scores was 4e-8 to 9e-8 larger without it. Over 60 sets of hypotheses within
// 0.005 rad and 5 cm of the current pose the rms error of the scores is 0.93 to 1.00
// of what it was with the projection in FP32 (Fisk): 1.01 to 1.09 on the driving scenes,
// 0.89 to 1.04 on the others; farther away single pixels beside the camera plane decide,
// either way.
constexpr double kScUntruncate = 1.0 + 4.3e-8;

// Sixteen bytes i < kScHypChunks of hypothesis h's operand row set to zero: a_z = U = V = 0 for
// every pixel. A pair of hypotheses shares a reciprocal, so with an odd count the row after
// the last one enters its score and may not hold what an earlier frame left there.
constexpr int kScHypChunks = 20;

__device__ __forceinline__ void clear_hyp_operand(unsigned char* base, int h, int i)
{
    unsigned char* d = base + (size_t)(h / kScStageHyps) * kScStageBytes + ((h % kScStageHyps) / 8) * 128 + (h % 8) * 16;
    if (i < 12) d += i / 4 * (kScStageHyps * 16) + i % 4 * kScHypSBlock;
    else d += (i < 16 ? kScHypUOff : kScHypVOff) + i % 4 * kScHypXBlock;
    *reinterpret_cast<uint4*>(d) = make_uint4(0u, 0u, 0u, 0u);
}

// Pixel chunks for a frame whose `groups` groups of hypotheses are fewer than a full
// frame's, by one converged warp: of 1 .. most chunks the number with the shortest
// schedule, as the host chooses it for full frames (rounds of the work items on the SMs times
// an item's tiles plus one and a half, the cost of starting and flushing an item). With
// the full frame's chunks a call with one group of S = 8192 left seven of eight SMs
// idle: 184 us a call for one hypothesis over 1242 x 375 pixels, now 124 (with its copies).
__device__ __forceinline__ int chunks_for_groups(int groups, int tiles, int most, int sms)
{
    const int lane = threadIdx.x & 31;
    most = min(most, tiles);
    unsigned best = 0xffffffffu;
    int at = 1;
    for (int c = lane + 1; c <= most; c += 32) {
        const unsigned cost = (unsigned)((groups * c + sms - 1) / sms) * (2u * (unsigned)((tiles + c - 1) / c) + 3u);
        if (cost < best) {
            best = cost;
            at = c;
        }
    }
    const unsigned least = __reduce_min_sync(0xffffffffu, best);
    return (int)__reduce_min_sync(0xffffffffu, best == least ? (unsigned)at : 0xffffffffu);
}

// Values beyond this size in a hypothesis's a_z coefficients or a pixel's x, y,
// w send a frame to the scoring's path without shared reciprocals: below it
// the product of two (1 + a_z) stays under 2^124.
constexpr float kScWild = 1073741824.f;                  // 2^30

// Operand row of hypothesis h from its scaled form (E, t) and the frame's reference
// pose (E0, t0), both FP64, by a quad of lanes: lane r < 3 is given row r, {E_r0, E_r1,
// E_r2, t_r}, and lane 3 row 2 again. Rows 0 and 1 make U's and V's coefficients, row 2
// those of a_z, which U and V need too. A warp issues an FP64 instruction every ~54
// cycles, so a lane per hypothesis would take three times as long. True in the lane
// that finds the hypothesis wild.
__device__ __forceinline__ bool write_hyp_operand(unsigned char* base, int h, const double* e, const double* e0)
{
    const int lane = threadIdx.x & 31, r = lane & 3;
    const unsigned quad = 0xfu << (lane & 28);
    const bool az = r >= 2;
    auto cut = [&](double v, double v0) {
        double d = az ? v - v0 : v0 - v;
        d *= kScUntruncate;
        const float hi = (float)d;
        return slice3(hi, (float)(d - (double)hi));
    };
    const Slice3 c[3] = {cut(e[0], e0[0]), cut(e[1], e0[1]), cut(e[3], e0[3])};      // of x, y, w
    const Slice3 c1 = cut(e[2], e0[2]);
    bool wild = false;
#pragma unroll
    for (int i = 0; i < 4; ++i) wild |= !(fabs(e[i]) < (double)kScWild) || !(fabs(e0[i]) < (double)kScWild);
    // row 2's slices to all lanes
    Slice3 z[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const Slice3& own = i < 3 ? c[i] : c1;
        const unsigned hm = (unsigned)__bfloat16_as_ushort(own.h) | (unsigned)__bfloat16_as_ushort(own.m) << 16;
        const unsigned a = __shfl_sync(quad, hm, 2, 4), b = __shfl_sync(quad, (unsigned)__bfloat16_as_ushort(own.l), 2, 4);
        z[i].h = __ushort_as_bfloat16((unsigned short)(a & 0xffffu));
        z[i].m = __ushort_as_bfloat16((unsigned short)(a >> 16));
        z[i].l = __ushort_as_bfloat16((unsigned short)b);
    }
    if (r == 3) return false;
    __align__(16) __nv_bfloat16 o[32];
    unsigned char* d = base + (size_t)(h / kScStageHyps) * kScStageBytes + ((h % kScStageHyps) / 8) * 128 + (h % 8) * 16;
    auto put = [&](unsigned char* dst, int stride) {
#pragma unroll
        for (int q = 0; q < 4; ++q) *reinterpret_cast<uint4*>(dst + q * stride) = *reinterpret_cast<const uint4*>(o + 8 * q);
    };
    hyp_block_s(c, c1, az, o);
    put(d + r * kScStageHyps * 16, kScHypSBlock);
    if (!az) {
        hyp_block_x(z, c, c1, o);
        put(d + (r == 0 ? kScHypUOff : kScHypVOff), kScHypXBlock);
    }
    return az && wild;
}

}  // namespace vd
