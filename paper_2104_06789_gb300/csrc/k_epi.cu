// Epipolar bootstrap of T_1 (Sec. 5.3 and Table 1: T_1 from the epipolar
// geometry of X_1 with a least-median-of-squares estimator).
//
//  1. k_epi_records: per pixel, the calibrated correspondence of X_1 as
//     {m0x, m0y, u/fx, v/fy} (FP32), m0 = K^-1 [x y 1]; NaN marks a pixel whose
//     flow target leaves I_1 (the test and the values are those of FP64).
//  2. k_epi_samples: eight lanes per minimal sample: 8 Philox-drawn pixels,
//     the 8-point essential matrix (null vector of the 8 x 9 system by Gaussian
//     elimination with complete pivoting, FP64), its projection onto the
//     essential matrices (eigen-decomposition of E^T E by Jacobi rotations),
//     and a scoring form: the decomposition [t]x R with the smaller rotation,
//     as Q = R - I and unit t in FP32.
//  3. The exact lower median of every valid sample's Sampson errors over all valid
//     pixels: k_epi_bracket brackets it from a regular subset of the pixels,
//     k_epi_count counts the errors below the bracket and collects those inside
//     it over all pixels, k_epi_median selects among these (and, should the bracket
//     have missed, by radix passes over all pixels). The Sampson error is evaluated
//     without cancellation: with m1 = m0 + d (d = flow / f, third component 0)
//     and R m0 = m0 + Q m0, the epipolar residual is
//         t . (m0 x d + (Q m0) x m1),
//     a sum of small terms, where m1^T E m0 would cancel O(1) products.
//     The last block takes the smallest median (lowest sample on ties).
//  4. Reweighted least squares: inliers of the winner (error <= (2.5 s)^2,
//     s = 1.4826 (1 + 5 / (n - 8)) sqrt(median)), A^T A of their rows
//     m1 (x) m0 in FP64 (per-block partials reduced in a fixed order), its
//     smallest eigenvector by inverse iteration, projected again.
//  5. The four decompositions; k_epi_cheirality counts the valid pixels whose
//     triangulated depth is positive in both cameras; the first candidate with
//     the largest count gives T_1, with |t| = the caller's baseline.
#include <cmath>

#include "voldor_internal.cuh"

namespace vd {

constexpr int kEpiSampleBlock = 64;
constexpr int kEpiSamplesPerBlock = 8;      // samples per histogram block
constexpr int kEpiBins = 2048;
constexpr int kEpiThreads = 256;

// ---------------------------------------------------------------------------
// 1. Records (and the count of valid pixels into info[2])
// ---------------------------------------------------------------------------
// 0 <= i + f <= last with the sum rounded to FP64, as the samples test it. A sum of
// an integer and an FP32 number keeps its sign when it is rounded, and one that is
// at most `last` stays so; what FP32 leaves open is an f just above last - i.
__device__ __forceinline__ bool target_inside(int i, float f, int last)
{
    const float c = (float)(last - i);
    if (!(f >= -(float)i)) return false;
    if (f <= c) return true;
    return f <= c + 1.f && (double)i + (double)f <= (double)last;
}

// (float)((double)f / fd) without an FP64 division where the FP32 result is beyond
// doubt: f times the float-float reciprocal has a relative error below 2^-43.
__device__ __forceinline__ float quotient32(float f, float inv_hi, float inv_lo, double fd)
{
    const float q = f * inv_hi;
    const float l = fmaf(f, inv_lo, fmaf(f, inv_hi, -q)), err = fabsf(q) * 0x1p-40f;
    const float below = __fadd_rn(q, l - err), above = __fadd_rn(q, l + err);
    if (below == above && (fabsf(q) > 1e-20f || f == 0.f)) return below;
    return (float)((double)f / fd);
}

// A warp takes 32 columns of kEpiRecRows rows: the FP64 divisions of m0 are one per
// column and one per row of the tile, not two per pixel (four with the flow's, which
// FP32 pairs replace): 52.5 -> 11.5 us at 1242 x 375.
constexpr int kEpiRecRows = 8, kEpiRecWarps = 8;

__global__ void __launch_bounds__(32 * kEpiRecWarps) k_epi_records(DevParams p, DevState s, EpiState e)
{
    __shared__ int inside_s[kEpiRecWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int x = blockIdx.x * 32 + lane, y0 = (blockIdx.y * kEpiRecWarps + warp) * kEpiRecRows;
    const float m0x = (float)(((double)x - p.cxd) / p.fxd);
    const float m0y_l = lane < kEpiRecRows ? (float)(((double)(y0 + lane) - p.cyd) / p.fyd) : 0.f;
    int inside = 0;
#pragma unroll
    for (int k = 0; k < kEpiRecRows; ++k) {
        const int y = y0 + k;
        const float m0y = __shfl_sync(0xffffffffu, m0y_l, k);
        const bool in_image = x < p.W && y < p.H;
        bool ok = false;
        if (in_image) {
            const size_t j = (size_t)y * p.W + x;
            const float2 f = load_flow(s.flows, p.flow_f16, j);
            ok = target_inside(x, f.x, p.W - 1) && target_inside(y, f.y, p.H - 1);
            float4 r = make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
            if (ok)
                r = make_float4(m0x, m0y, quotient32(f.x, p.kdf[8], p.kdf[9], p.fxd),
                                quotient32(f.y, p.kdf[10], p.kdf[11], p.fyd));
            e.rec[j] = r;
        }
        inside += __popc(__ballot_sync(0xffffffffu, ok));
    }
    if (lane == 0) inside_s[warp] = inside;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kEpiRecWarps; ++w) inside += inside_s[w];
        if (inside) atomicAdd(reinterpret_cast<unsigned long long*>(e.info + 2), (unsigned long long)inside);
    }
}

// ---------------------------------------------------------------------------
// FP64 helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void cross3d(const double* a, const double* b, double* o)
{
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ bool unit3d(double* a)
{
    const double n = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
    if (!(n > 0.0)) return false;
    a[0] /= n; a[1] /= n; a[2] /= n;
    return true;
}

// Symmetric 3 x 3 eigen-decomposition by cyclic Jacobi rotations (two-sided):
// A (row-major) is overwritten; columns of V are the eigenvectors, d the values.
__device__ void sym3_eigen(double* A, double* d, double* V)
{
    for (int i = 0; i < 9; ++i) V[i] = (i % 4 == 0) ? 1.0 : 0.0;
    for (int sweep = 0; sweep < 30; ++sweep) {
        const double off = A[1] * A[1] + A[2] * A[2] + A[5] * A[5];
        const double dia = A[0] * A[0] + A[4] * A[4] + A[8] * A[8];
        if (!(off > 1e-32 * dia)) break;
        for (int pq = 0; pq < 3; ++pq) {
            const int pp = pq == 2 ? 1 : 0, qq = pq == 0 ? 1 : 2;
            const double apq = A[pp * 3 + qq];
            if (apq == 0.0) continue;
            const double th = (A[qq * 3 + qq] - A[pp * 3 + pp]) / (2.0 * apq);
            const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            const double c = 1.0 / sqrt(t * t + 1.0), sn = t * c;
            for (int k = 0; k < 3; ++k) {
                const double akp = A[k * 3 + pp], akq = A[k * 3 + qq];
                A[k * 3 + pp] = c * akp - sn * akq;
                A[k * 3 + qq] = sn * akp + c * akq;
            }
            for (int k = 0; k < 3; ++k) {
                const double apk = A[pp * 3 + k], aqk = A[qq * 3 + k];
                A[pp * 3 + k] = c * apk - sn * aqk;
                A[qq * 3 + k] = sn * apk + c * aqk;
            }
            for (int k = 0; k < 3; ++k) {
                const double vkp = V[k * 3 + pp], vkq = V[k * 3 + qq];
                V[k * 3 + pp] = c * vkp - sn * vkq;
                V[k * 3 + qq] = sn * vkp + c * vkq;
            }
        }
    }
    d[0] = A[0]; d[1] = A[4]; d[2] = A[8];
}

// Projection onto the essential matrices, E = U diag(1, 1, 0) V^T with
// det U = det V = +1, from the eigenvectors of Ein^T Ein. False if rank < 2.
// Kept out of line: inlined into k_epi_samples by nvcc 13.0 it returned false
// for valid input, while the same code called out of line (and a line-by-line
// NumPy replay) returns the correct projection; the cause was not found.
__device__ __noinline__ bool essential_project(const double* Ein, double* E, double* U, double* V)
{
    double A[9], d[3], Q[9];
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 3; ++b)
            A[a * 3 + b] = Ein[a] * Ein[b] + Ein[3 + a] * Ein[3 + b] + Ein[6 + a] * Ein[6 + b];
    sym3_eigen(A, d, Q);
    int o0 = 0, o1 = 1, o2 = 2;                       // descending order of d
    if (d[o0] < d[o1]) { const int t = o0; o0 = o1; o1 = t; }
    if (d[o1] < d[o2]) { const int t = o1; o1 = o2; o2 = t; }
    if (d[o0] < d[o1]) { const int t = o0; o0 = o1; o1 = t; }
    double v[3][3], u[3][3];
    const int oi[2] = {o0, o1};
    for (int i = 0; i < 2; ++i)
        for (int k = 0; k < 3; ++k) v[i][k] = Q[k * 3 + oi[i]];
    cross3d(v[0], v[1], v[2]);
    for (int i = 0; i < 2; ++i) {
        for (int r = 0; r < 3; ++r) u[i][r] = Ein[r * 3 + 0] * v[i][0] + Ein[r * 3 + 1] * v[i][1] + Ein[r * 3 + 2] * v[i][2];
        if (!unit3d(u[i])) return false;
    }
    // u_1 is orthogonal to u_0 in exact arithmetic; re-orthogonalise
    const double dd = u[0][0] * u[1][0] + u[0][1] * u[1][1] + u[0][2] * u[1][2];
    for (int r = 0; r < 3; ++r) u[1][r] -= dd * u[0][r];
    if (!unit3d(u[1])) return false;
    cross3d(u[0], u[1], u[2]);
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            U[r * 3 + c] = u[c][r];
            V[r * 3 + c] = v[c][r];
            E[r * 3 + c] = u[0][r] * v[0][c] + u[1][r] * v[1][c];
        }
    return true;
}

// R = U W V^T (a = 0) or U W^T V^T (a = 1), W = [[0,-1,0],[1,0,0],[0,0,1]].
__device__ void rot_candidate(const double* U, const double* V, int a, double* R)
{
    // U W: columns (u1, -u0, u2); U W^T: columns (-u1, u0, u2)
    double UW[9];
    for (int r = 0; r < 3; ++r) {
        UW[r * 3 + 0] = a == 0 ? U[r * 3 + 1] : -U[r * 3 + 1];
        UW[r * 3 + 1] = a == 0 ? -U[r * 3 + 0] : U[r * 3 + 0];
        UW[r * 3 + 2] = U[r * 3 + 2];
    }
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c)
            R[r * 3 + c] = UW[r * 3 + 0] * V[c * 3 + 0] + UW[r * 3 + 1] * V[c * 3 + 1] + UW[r * 3 + 2] * V[c * 3 + 2];
}

// Scoring form of an essential matrix: the rotation candidate with the larger
// trace (the smaller angle) as Q = R - I, and t = u_2.
__device__ void scoring_form(const double* U, const double* V, float* f)
{
    double Ra[9], Rb[9];
    rot_candidate(U, V, 0, Ra);
    rot_candidate(U, V, 1, Rb);
    const double* R = (Ra[0] + Ra[4] + Ra[8] >= Rb[0] + Rb[4] + Rb[8]) ? Ra : Rb;
    for (int i = 0; i < 9; ++i) f[i] = (float)(R[i] - ((i % 4 == 0) ? 1.0 : 0.0));
    for (int r = 0; r < 3; ++r) f[9 + r] = (float)U[r * 3 + 2];
}

// ---------------------------------------------------------------------------
// 2. Minimal samples
// ---------------------------------------------------------------------------
// Eight lanes per sample, a lane per correspondence and row of the 8 x 9 system.
// What bounds it is the chain of one sample's FP64 instructions (~75 cycles each), so
// a step of the elimination costs a row's update and a search over the lanes instead
// of the whole matrix: on one thread per sample, the matrix in local memory, 512
// samples took 119 us; now 75 us, most of it the projection's Jacobi rotations.
// Every entry sees the operations of row-by-row elimination in the same order.
constexpr int kEpiSampleLanes = 8;

__device__ void epi_sample(const DevParams& p, const DevState& s, const EpiState& e, int m)
{
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31, row = lane & 7;
    const U64x4 rnd = philox4x64_10((uint64_t)m, (uint64_t)(row >> 2), 0, (uint64_t)kStreamEpi, p.seed, p.window_id);
    uint64_t draw = rnd.v[0];
#pragma unroll
    for (int i = 1; i < 4; ++i)
        if ((row & 3) == i) draw = rnd.v[i];
    const long long j = (long long)__umul64hi(draw, (uint64_t)p.N);
    bool dup = false;
#pragma unroll
    for (int i = 1; i < 8; ++i) dup |= __shfl_xor_sync(kAll, j, i) == j;
    const int x = (int)(j % p.W), y = (int)(j / p.W);
    const float2 f = load_flow(s.flows, p.flow_f16, (size_t)j);
    const double u = (double)x + (double)f.x, v = (double)y + (double)f.y;
    const bool inside = u >= 0.0 && u <= (double)(p.W - 1) && v >= 0.0 && v <= (double)(p.H - 1);
    const unsigned group = 0xffu << (lane & 24);
    const unsigned dups = __ballot_sync(kAll, dup), insides = __ballot_sync(kAll, inside);
    int why = dups & group ? -1 : (~insides & group ? -2 : 1);
    // (lanes of a sample agree on `why`; the warp's samples run the same code, a
    // rejected one on values that go nowhere)
    const double m0[3] = {((double)x - p.cxd) / p.fxd, ((double)y - p.cyd) / p.fyd, 1.0};
    const double m1[3] = {(u - p.cxd) / p.fxd, (v - p.cyd) / p.fyd, 1.0};
    double A[9];
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
        for (int c = 0; c < 3; ++c) A[r * 3 + c] = m1[r] * m0[c];

    // Gaussian elimination with complete pivoting. Rows stay in their lanes: `pos` is
    // the row's place, `holder` and `col` (four bits each) the lane of each place
    // that is done and the order of the columns.
    int pos = row;
    unsigned holder = 0;
    unsigned long long col = 0x876543210ull;
    double piv0 = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        double best = pos >= k ? -1.0 : -2.0;
        int bc = k, at = pos, from = row;
        if (pos >= k) {
#pragma unroll
            for (int c = k; c < 9; ++c)
                if (fabs(A[c]) > best) { best = fabs(A[c]); bc = c; }
        }
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
            const double ob = __shfl_xor_sync(kAll, best, o);
            const int packed = __shfl_xor_sync(kAll, bc | at << 8 | from << 16, o), oat = packed >> 8 & 255;
            if (ob > best || (ob == best && oat < at)) { best = ob; bc = packed & 255; at = oat; from = packed >> 16; }
        }
        if (k == 0) piv0 = best;
        if (why == 1 && (!(best > 1e-12 * piv0) || !(best > 0.0))) why = -3;
        if (pos == k) pos = at;                       // rows k and `at` change places
        if (row == from) pos = k;
        holder |= (unsigned)from << (4 * k);
#pragma unroll
        for (int c = k + 1; c < 9; ++c)
            if (c == bc) { const double t = A[k]; A[k] = A[c]; A[c] = t; }
        const unsigned long long d = (col >> 4 * k ^ col >> 4 * bc) & 15;
        col ^= d << 4 * k;
        col ^= d << 4 * bc;
        const double inv = 1.0 / __shfl_sync(kAll, A[k], from, 8);
        const double fr = pos > k ? A[k] * inv : 0.0;
#pragma unroll
        for (int c = k + 1; c < 9; ++c) {
            const double pc = __shfl_sync(kAll, A[c], from, 8);
            if (fr != 0.0) A[c] = fma(-fr, pc, A[c]);
        }
    }
    double z[9];
    z[8] = 1.0;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
        double acc = 0.0;
#pragma unroll
        for (int c = k + 1; c < 9; ++c) acc = fma(A[c], z[c], acc);
        z[k] = __shfl_sync(kAll, -acc / A[k], (int)(holder >> (4 * k)) & 7, 8);
    }
    if (row != 0 || m >= e.M) return;
    double Ev[9], E[9], U[9], V[9];
    double nn = 0.0;
    for (int c = 0; c < 9; ++c) nn += z[c] * z[c];
    nn = 1.0 / sqrt(nn);
    for (int c = 0; c < 9; ++c) Ev[(int)(col >> 4 * c) & 15] = z[c] * nn;
    if (why == 1 && !essential_project(Ev, E, U, V)) why = -4;
    e.valid[m] = why;
    float* form = e.form + (size_t)m * 12;
    if (why == 1) {
        for (int i = 0; i < 9; ++i) {
            e.E[(size_t)m * 9 + i] = E[i];
            e.UV[(size_t)m * 18 + i] = U[i];
            e.UV[(size_t)m * 18 + 9 + i] = V[i];
        }
        scoring_form(U, V, form);
    } else {
        for (int i = 0; i < 9; ++i) e.E[(size_t)m * 9 + i] = 0.0;
        for (int i = 0; i < 12; ++i) form[i] = 0.f;
        e.median[m] = __int_as_float(0x7f800000);
    }
}

// The last block to finish lists the valid samples in order (the median passes
// then work on full groups of them: of a fast forward motion's samples most hold a
// pixel whose target leaves the image).
__global__ void __launch_bounds__(kEpiSampleBlock) k_epi_samples(DevParams p, DevState s, EpiState e)
{
    const int m = (blockIdx.x * blockDim.x + threadIdx.x) / kEpiSampleLanes;
    if ((m & ~3) < e.M) epi_sample(p, s, e, m);        // whole warps; samples past M are not written
    __threadfence();
    __shared__ bool last;
    __shared__ int wsum[kEpiSampleBlock / 32];
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(e.done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int base = 0;
    for (int m0 = 0; m0 < e.M; m0 += kEpiSampleBlock) {
        const int i = m0 + threadIdx.x;
        const bool ok = i < e.M && __ldcg(e.valid + i) > 0;
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        if (lane == 0) wsum[warp] = __popc(bal);
        __syncthreads();
        int before = base, all = 0;
        for (int w = 0; w < kEpiSampleBlock / 32; ++w) {
            if (w < warp) before += wsum[w];
            all += wsum[w];
        }
        if (ok) e.list[before + __popc(bal & ((1u << lane) - 1u))] = i;
        base += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) *e.n_list = base;
}

// ---------------------------------------------------------------------------
// 3. Sampson error (FP32, cancellation-free) and radix selection of the median
// ---------------------------------------------------------------------------
// Numerator and denominator: the error is e2 / den, +inf where den is not positive
// or the quotient no number.
__device__ __forceinline__ void sampson_parts(const float* F, float4 r, float& e2, float& den)
{
    const float m0x = r.x, m0y = r.y, dx = r.z, dy = r.w;
    const float m1x = m0x + dx, m1y = m0y + dy;
    const float q0 = fmaf(F[0], m0x, fmaf(F[1], m0y, F[2]));
    const float q1 = fmaf(F[3], m0x, fmaf(F[4], m0y, F[5]));
    const float q2 = fmaf(F[6], m0x, fmaf(F[7], m0y, F[8]));
    const float tx = F[9], ty = F[10], tz = F[11];
    // c = m0 x d + q x m1
    const float cx = -dy + (q1 - q2 * m1y);
    const float cy = dx + (q2 * m1x - q0);
    const float cz = fmaf(m0x, dy, -m0y * dx) + fmaf(q0, m1y, -q1 * m1x);
    const float e = fmaf(tx, cx, fmaf(ty, cy, tz * cz));
    // E m0 = t x (m0 + q)
    const float rx = m0x + q0, ry = m0y + q1, rz = 1.f + q2;
    const float a0 = fmaf(ty, rz, -tz * ry), a1 = fmaf(tz, rx, -tx * rz);
    // E^T m1 = -R^T (t x m1), R = I + Q
    const float w0 = fmaf(ty, 1.f, -tz * m1y), w1 = fmaf(tz, m1x, -tx), w2 = fmaf(tx, m1y, -ty * m1x);
    const float b0 = w0 + fmaf(F[0], w0, fmaf(F[3], w1, F[6] * w2));
    const float b1 = w1 + fmaf(F[1], w0, fmaf(F[4], w1, F[7] * w2));
    den = fmaf(a0, a0, fmaf(a1, a1, fmaf(b0, b0, b1 * b1)));
    e2 = e * e;
}

__device__ __forceinline__ float sampson_ratio(float e2, float den)
{
    const float d = e2 / den;
    return (den > 0.f && d == d) ? d : __int_as_float(0x7f800000);
}

__device__ __forceinline__ float sampson32(const float* F, float4 r)
{
    float e2, den;
    sampson_parts(F, r, e2, den);
    return sampson_ratio(e2, den);
}

constexpr int kEpiPix = 4;                                   // pixels per thread of a work item
constexpr int kEpiItemPix = kEpiThreads * kEpiPix;           // 1024
// Loads a group's scoring forms; the samples of group g are list[8 g ...].
__device__ __forceinline__ int epi_load_group(const EpiState& e, int g, int n, float (*F)[12], int* id)
{
    const int cnt = min(kEpiSamplesPerBlock, n - g * kEpiSamplesPerBlock);
    if ((int)threadIdx.x < cnt * 12) {
        const int sm = threadIdx.x / 12, q = threadIdx.x % 12, m = e.list[g * kEpiSamplesPerBlock + sm];
        F[sm][q] = e.form[(size_t)m * 12 + q];
        if (q == 0) id[sm] = m;
    }
    return cnt;
}

// The bin of a block's shared histogram that holds rank `rank`, and the rank inside
// it (all threads get both); false if the counts do not reach the rank.
__device__ __forceinline__ bool epi_pick(const unsigned* h, int bins, unsigned rank, unsigned* ws, unsigned& bin, unsigned& rest)
{
    __shared__ unsigned out[2];
    const int per = (bins + blockDim.x - 1) / blockDim.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned mine = 0;
    for (int i = 0; i < per; ++i) {
        const int b = threadIdx.x * per + i;
        if (b < bins) mine += h[b];
    }
    unsigned incl = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) ws[warp] = incl;
    if (threadIdx.x == 0) out[0] = 0xffffffffu;
    __syncthreads();
    unsigned cum = incl - mine;
    for (int w = 0; w < warp; ++w) cum += ws[w];
    for (int i = 0; i < per; ++i) {
        const int b = threadIdx.x * per + i;
        const unsigned c = b < bins ? h[b] : 0u;
        if (rank >= cum && rank < cum + c) { out[0] = (unsigned)b; out[1] = rank - cum; }
        cum += c;
    }
    __syncthreads();
    bin = out[0];
    rest = out[1];
    __syncthreads();
    return bin != 0xffffffffu;
}

// The value of rank `rank` among n bit patterns in [lo, lo + span), by the block's radix
// passes of 11 bits from the top of the span; false if they do not hold the rank.
__device__ bool epi_select(const unsigned* v, unsigned n, unsigned lo, unsigned span, unsigned rank, unsigned* h, unsigned* ws,
                           unsigned& bits)
{
    unsigned from = lo, width = span, bin;
    bool ok = true;
    while (width > 1 && ok) {
        const int shift = max(0, 32 - __clz(width - 1) - 11);
        for (int i = threadIdx.x; i < kEpiBins; i += blockDim.x) h[i] = 0;
        __syncthreads();
        for (unsigned i = threadIdx.x; i < n; i += blockDim.x) {
            const unsigned o = v[i] - from;
            if (o < width) atomicAdd(&h[o >> shift], 1u);
        }
        __syncthreads();
        ok = epi_pick(h, kEpiBins, rank, ws, bin, rank);
        from += bin << shift;
        width = 1u << shift;
    }
    bits = from;
    return ok;
}

// Pixels of the second subset, from which k_epi_bracket narrows a bracket that may hold more
// errors than `cap`: four and a half standard deviations of so many then are three
// quarters of `cap`, as long as the 3.5 % of them inside the first bracket fit too.
__device__ __forceinline__ int epi_second_subset(int N, int cap)
{
    const double n = 6.0 * (double)N / (double)cap;
    return (int)fmin(fmin(n * n, 24.0 * (double)cap), (double)N);
}

// Bracket of the median from a subset of the pixels, one block per valid sample:
// one pixel of every `step`, at a place that varies (all pixels of a small image),
// 16384 errors in registers at most; the subset's ranks four and a half standard
// deviations of a binomial count below and above its median are selected exactly
// by radix passes. Between them lie about 3.5 % of all errors; a bracket that
// misses costs time (k_epi_median), not exactness. Bound by the latency of the
// strided record loads and of the six scans between barriers.
//
// From 1.4 million pixels on 3.5 % of them come near the room for the collected errors, and
// beyond 1.87 million every sample went to the passes over all pixels (1920 x 1080, 64
// samples: 2.7 ms, 1.8 with three histograms over all pixels). There the block goes over
// a second, larger subset, keeps its errors inside the first bracket and selects the
// same ranks' bounds among them: now 0.57 ms.
constexpr int kEpiSubThreads = 512, kEpiSubPer = 32;

__global__ void __launch_bounds__(kEpiSubThreads, 2) k_epi_bracket(DevParams p, EpiState e)
{
    __shared__ unsigned h[2][kEpiBins], ws[kEpiSubThreads / 32];
    __shared__ __align__(16) float F[12];
    if ((int)blockIdx.x >= *e.n_list) return;
    const int q = blockIdx.x;
    if (threadIdx.x < 12) F[threadIdx.x] = e.form[(size_t)e.list[q] * 12 + threadIdx.x];
    for (int i = threadIdx.x; i < kEpiBins; i += blockDim.x) h[0][i] = 0;
    __syncthreads();
    const int step = (p.N + kEpiSubThreads * kEpiSubPer - 1) / (kEpiSubThreads * kEpiSubPer), n_sub = p.N / step;
    constexpr unsigned kNone = 0xffffffffu;
    unsigned v[kEpiSubPer], mine = 0;
#pragma unroll
    for (int i = 0; i < kEpiSubPer; ++i) {
        const int k = i * kEpiSubThreads + threadIdx.x;
        v[i] = kNone;
        if (k < n_sub) {
            const float4 r = e.rec[(size_t)k * step + (unsigned)(k * 5) % (unsigned)step];
            if (r.x == r.x) {
                v[i] = __float_as_uint(sampson32(F, r));
                ++mine;
                atomicAdd(&h[0][v[i] >> 21], 1u);
            }
        }
    }
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
    __shared__ unsigned total_s;
    if (threadIdx.x == 0) total_s = 0;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) atomicAdd(&total_s, mine);
    __syncthreads();
    const unsigned total = total_s;
    if (total == 0) {
        if (threadIdx.x == 0) e.lo[q] = e.hi[q] = 0u;
        return;
    }
    const float mid = 0.5f * (float)total, dev = step > 1 ? 2.25f * sqrtf((float)total) + 2.f : 1.f;
    unsigned rank[2] = {mid > dev ? (unsigned)(mid - dev) : 0u, min((unsigned)(mid + dev), total - 1u)}, prefix[2];
    for (int r = 0; r < 2; ++r) epi_pick(h[0], 1024, rank[r], ws, prefix[r], rank[r]);
    for (int level = 0; level < 2; ++level) {
        const int shift = level == 0 ? 10 : 0, top = level == 0 ? 21 : 10, bins = level == 0 ? 2048 : 1024;
        for (int i = threadIdx.x; i < bins; i += blockDim.x) h[0][i] = h[1][i] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kEpiSubPer; ++i)
#pragma unroll
            for (int r = 0; r < 2; ++r)
                if (v[i] != kNone && (v[i] >> top) == prefix[r]) atomicAdd(&h[r][(v[i] >> shift) & (bins - 1)], 1u);
        __syncthreads();
        for (int r = 0; r < 2; ++r) {
            unsigned bin;
            epi_pick(h[r], bins, rank[r], ws, bin, rank[r]);
            prefix[r] = (prefix[r] << (top - shift)) | bin;
        }
    }
    unsigned lo = prefix[0], hi = prefix[1] + 1u;
    if (step > 1 && (float)p.N * (2.f * dev) > 0.75f * (float)e.cap * (float)n_sub && hi - lo > 1) {
        const int step2 = p.N / epi_second_subset(p.N, e.cap), n2 = p.N / step2;
        unsigned* v2 = e.found + (size_t)q * e.cap;          // free until k_epi_count
        __shared__ unsigned count[3];                        // errors of the subset, below the bracket, inside it
        if (threadIdx.x < 3) count[threadIdx.x] = 0;
        __syncthreads();
        unsigned all = 0, under = 0;
        for (int k = threadIdx.x; k < n2; k += kEpiSubThreads) {
            const float4 r = e.rec[(size_t)k * step2 + (unsigned)(k * 5) % (unsigned)step2];
            if (r.x != r.x) continue;
            const unsigned bits = __float_as_uint(sampson32(F, r));
            ++all;
            if (bits < lo) ++under;
            else if (bits < hi) {
                const unsigned at = atomicAdd(&count[2], 1u);
                if (at < (unsigned)e.cap) v2[at] = bits;
            }
        }
        all = __reduce_add_sync(0xffffffffu, all);
        under = __reduce_add_sync(0xffffffffu, under);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&count[0], all);
            atomicAdd(&count[1], under);
        }
        __syncthreads();
        const unsigned in = count[2];
        const double mid2 = 0.5 * (double)count[0], dev2 = 2.25 * sqrt((double)count[0]) + 2.0;
        // a bound that lies outside the first bracket leaves that side as it is
        const double r0 = floor(mid2 - dev2) - (double)count[1], r1 = ceil(mid2 + dev2) - (double)count[1];
        if (in <= (unsigned)e.cap && r0 < (double)in && r1 >= 0.0) {
            const unsigned from = lo, span = hi - lo;
            unsigned b;
            if (r0 >= 0.0 && epi_select(v2, in, from, span, (unsigned)r0, h[0], ws, b)) lo = b;
            if (r1 < (double)in && epi_select(v2, in, from, span, (unsigned)r1, h[0], ws, b)) hi = b + 1u;
        }
    }
    if (threadIdx.x == 0) {
        e.lo[q] = lo;
        e.hi[q] = hi;
    }
}

// One pass over all pixels: per sample, the errors below its bracket are counted
// and those inside it collected. An error is compared without the division, e2
// against the edge times den, unless it lies within 2^-20 of an edge or inside the
// bracket (a few percent of the pairs); only then is the rounded quotient formed.
// The 1e-30 keeps products that round as denormals out of the short way.
// Four pixels per thread share a sample's form. What bounds it: the ~45 FP32
// instructions of a pair. 512 samples over 1242 x 375 pixels: three radix passes
// over all pixels, with a division and a shared-memory atomic per pair and pass,
// took 735 us; bracket, count and selection take 45 + 157 + 18 us.
__global__ void __launch_bounds__(kEpiThreads, 3) k_epi_count(DevParams p, EpiState e)
{
    __shared__ __align__(16) float F[kEpiSamplesPerBlock][12];
    __shared__ int id[kEpiSamplesPerBlock];
    __shared__ float edge[kEpiSamplesPerBlock][2];
    __shared__ unsigned lo_s[kEpiSamplesPerBlock], hi_s[kEpiSamplesPerBlock], below[kEpiSamplesPerBlock];
    __shared__ unsigned fill[kEpiSamplesPerBlock], base[kEpiSamplesPerBlock];
    __shared__ unsigned found[kEpiSamplesPerBlock][kEpiItemPix];
    const int n = *e.n_list, groups = (n + kEpiSamplesPerBlock - 1) / kEpiSamplesPerBlock;
    const int chunks = (p.N + kEpiItemPix - 1) / kEpiItemPix, lane = threadIdx.x & 31;
    for (int u = blockIdx.x; u < groups * chunks; u += gridDim.x) {
        const int g = u / chunks, j0 = (u % chunks) * kEpiItemPix, q0 = g * kEpiSamplesPerBlock;
        const int cnt = epi_load_group(e, g, n, F, id);
        if ((int)threadIdx.x < cnt) {
            lo_s[threadIdx.x] = e.lo[q0 + threadIdx.x];
            hi_s[threadIdx.x] = e.hi[q0 + threadIdx.x];
            edge[threadIdx.x][0] = __uint_as_float(lo_s[threadIdx.x]) * (1.f - 9.5367432e-7f);
            edge[threadIdx.x][1] = __uint_as_float(hi_s[threadIdx.x]) * (1.f + 9.5367432e-7f);
            below[threadIdx.x] = fill[threadIdx.x] = 0u;
        }
        __syncthreads();
        float4 r[kEpiPix];
#pragma unroll
        for (int i = 0; i < kEpiPix; ++i) {
            const int j = j0 + i * kEpiThreads + threadIdx.x;
            r[i] = j < p.N ? e.rec[j] : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
        }
        for (int sm = 0; sm < cnt; ++sm) {
            float f[12];
#pragma unroll
            for (int i = 0; i < 12; ++i) f[i] = F[sm][i];
            const float lo_m = edge[sm][0], hi_p = edge[sm][1];
            unsigned less = 0;
#pragma unroll
            for (int i = 0; i < kEpiPix; ++i) {
                float e2, den;
                sampson_parts(f, r[i], e2, den);
                if (e2 < fmaf(lo_m, den, -1e-30f)) {
                    ++less;
                } else if (!(e2 > fmaf(hi_p, den, 1e-30f)) && r[i].x == r[i].x) {
                    const unsigned bits = __float_as_uint(sampson_ratio(e2, den));
                    if (bits < lo_s[sm]) ++less;
                    else if (bits < hi_s[sm]) found[sm][atomicAdd(&fill[sm], 1u)] = bits;
                }
            }
            less = __reduce_add_sync(0xffffffffu, less);
            if (lane == 0 && less) atomicAdd(&below[sm], less);
        }
        __syncthreads();
        if ((int)threadIdx.x < cnt) {
            if (below[threadIdx.x]) atomicAdd(e.below + q0 + threadIdx.x, below[threadIdx.x]);
            base[threadIdx.x] = fill[threadIdx.x] ? atomicAdd(e.inside + q0 + threadIdx.x, fill[threadIdx.x]) : 0u;
        }
        __syncthreads();
        for (int sm = 0; sm < cnt; ++sm)
            for (unsigned i = threadIdx.x; i < fill[sm]; i += blockDim.x)
                if (base[sm] + i < (unsigned)e.cap && hi_s[sm] - lo_s[sm] > 1) e.found[(size_t)(q0 + sm) * e.cap + base[sm] + i] = found[sm][i];
        __syncthreads();
    }
}

// One block per valid sample: the exact median, rank (n - 1) / 2 of the valid
// pixels' errors, among the collected ones (radix passes over the bracket's bit
// patterns, 11 bits each; a bracket of one bit pattern is the median itself);
// where they do not hold it, radix passes over all pixels (11 + 11 + 10 bits).
constexpr int kEpiMedianThreads = 1024;

__device__ __forceinline__ void epi_median(const DevParams& p, const EpiState& e, int q)
{
    __shared__ unsigned h[kEpiBins], ws[kEpiMedianThreads / 32];
    __shared__ __align__(16) float F[12];
    const int m = e.list[q];
    const long long nv = e.info[2];
    if (nv == 0) {
        if (threadIdx.x == 0) e.median[m] = __int_as_float(0x7f800000);
        return;
    }
    const unsigned rank = (unsigned)((nv - 1) / 2), under = e.below[q], in = e.inside[q], lo = e.lo[q];
    const unsigned span = e.hi[q] - lo;                                // at most 2^31
    unsigned bits = 0, bin, rest;
    bool ok = rank >= under && rank - under < in && (in <= (unsigned)e.cap || span == 1);
    if (ok) ok = epi_select(e.found + (size_t)q * e.cap, in, lo, span, rank - under, h, ws, bits);
    if (!ok) {
        if (threadIdx.x < 12) F[threadIdx.x] = e.form[(size_t)m * 12 + threadIdx.x];
        unsigned prefix = 0;
        rest = rank;
        ok = true;
        for (int pass = 0; pass < 3 && ok; ++pass) {
            const int shift = pass == 0 ? 21 : (pass == 1 ? 10 : 0), width = pass == 2 ? 1024 : 2048;
            for (int i = threadIdx.x; i < kEpiBins; i += blockDim.x) h[i] = 0;
            __syncthreads();
            for (int j = threadIdx.x; j < p.N; j += blockDim.x) {
                const float4 r = e.rec[j];
                if (r.x != r.x) continue;
                const unsigned b = __float_as_uint(sampson32(F, r));
                if (pass == 0 || (b >> (pass == 1 ? 21 : 10)) == prefix) atomicAdd(&h[(b >> shift) & (width - 1)], 1u);
            }
            __syncthreads();
            ok = epi_pick(h, width, rest, ws, bin, rest);
            prefix = pass == 0 ? bin : (prefix << (pass == 1 ? 11 : 10)) | bin;
        }
        bits = ok ? prefix : 0x7f800000u;
    }
    if (threadIdx.x == 0) e.median[m] = __uint_as_float(bits);
}

// The last block to finish takes the winner: the smallest median, the lowest sample
// on ties.
__global__ void __launch_bounds__(kEpiMedianThreads, 2) k_epi_median(DevParams p, EpiState e)
{
    if ((int)blockIdx.x < *e.n_list) epi_median(p, e, blockIdx.x);
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(e.median_done, 1) == (int)gridDim.x - 1;
        __threadfence();
    }
    __syncthreads();
    if (!last) return;
    float best = __int_as_float(0x7f800000);
    int bi = 0x7fffffff;
    for (int m = threadIdx.x; m < e.M; m += blockDim.x) {
        const float v = __ldcg(e.median + m);
        if (v < best || (v == best && m < bi)) { best = v; bi = m; }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov < best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    __shared__ float wv[32];
    __shared__ int wi[32];
    if ((threadIdx.x & 31) == 0) { wv[threadIdx.x >> 5] = best; wi[threadIdx.x >> 5] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            if (wv[w] < best || (wv[w] == best && wi[w] < bi)) { best = wv[w]; bi = wi[w]; }
        const bool any = best < __int_as_float(0x7f800000);
        e.info[0] = any ? bi : -1;
    }
}

// ---------------------------------------------------------------------------
// 4. Reweighted least squares
// ---------------------------------------------------------------------------
// Sums of 32 values over the warp in 31 additions a lane: lane l gets value l's.
__device__ __forceinline__ double warp_sum32d(double (&v)[32])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int h = 16; h > 0; h >>= 1) {
        const bool up = lane & h;
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const double send = up ? v[i] : v[i + h], keep = up ? v[i + h] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
        }
    }
    return v[0];
}

// A^T A over the winner's inliers. Its 45 entries are 36 different sums, of a product
// of two of (x, y, 1) with a product of two of (u, v, 1): pixel and target relative to
// the principal point; the focal lengths are divided out of the sums. A lane stays in
// a column and walks kEpiAccRows rows, so it adds y^k {uu, uv, u, vv, v, 1} only,
// k = 0, 1, 2, and multiplies by x and x^2 at the end. What bounds it: FP64, two lanes
// a clock, 24 instructions a pixel where the 45 sums with their divisions took 120:
// 116 -> 44 us at 1242 x 375.
constexpr int kEpiAccRows = 16, kEpiAccWarps = 4, kEpiSums = 36;

__global__ void __launch_bounds__(32 * kEpiAccWarps) k_epi_refine_accum(DevParams p, DevState s, EpiState e)
{
    __shared__ float F[12];
    __shared__ float thr;
    __shared__ double ws[kEpiAccWarps][kEpiSums];
    const long long best = e.info[0];
    if (best < 0) return;
    if (threadIdx.x < 12) F[threadIdx.x] = e.form[best * 12 + threadIdx.x];
    if (threadIdx.x == 0) {
        const double n = (double)e.info[2];
        const double sc = 1.4826 * (1.0 + 5.0 / fmax(n - 8.0, 1.0)) * sqrt((double)e.median[best]);
        thr = (float)((2.5 * sc) * (2.5 * sc));
    }
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, tiles = (p.W + 31) / 32;
    const int item = blockIdx.x * kEpiAccWarps + warp;
    const int x = (item % tiles) * 32 + lane, y0 = (item / tiles) * kEpiAccRows;
    const double xc = (double)x - p.cxd;
    double a[3][5], sy = 0.0, syy = 0.0;
    int count = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 5; ++i) a[k][i] = 0.0;
    constexpr int kAhead = 4;
    for (int k0 = 0; k0 < kEpiAccRows; k0 += kAhead) {
        float4 r[kAhead];
        float2 f[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int y = y0 + k0 + k;
            const bool in_image = x < p.W && y < p.H;
            r[k] = in_image ? e.rec[(size_t)y * p.W + x] : make_float4(__int_as_float(0x7fc00000), 0.f, 0.f, 0.f);
            f[k] = in_image ? load_flow(s.flows, p.flow_f16, (size_t)y * p.W + x) : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            if (r[k].x != r[k].x || !(sampson32(F, r[k]) <= thr)) continue;
            const double y = (double)(y0 + k0 + k) - p.cyd, yy = y * y;
            const double u = xc + (double)f[k].x, v = y + (double)f[k].y;
            const double q[5] = {u * u, u * v, u, v * v, v};
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                a[0][i] += q[i];
                a[1][i] += y * q[i];
                a[2][i] += yy * q[i];
            }
            sy += y;
            syy += yy;
            ++count;
        }
    }
    const double n = (double)count, xx = xc * xc;
    double lo[32], hi[3];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const double s0 = i < 5 ? a[0][i % 5] : n, s1 = i < 5 ? a[1][i % 5] : sy, s2 = i < 5 ? a[2][i % 5] : syy;
        lo[i] = xx * s0;
        lo[6 + i] = xc * s1;
        lo[12 + i] = xc * s0;
        lo[18 + i] = s2;
        lo[24 + i] = s1;
        if (i < 2) lo[30 + i] = s0;
        else if (i < 5) hi[i - 2] = s0;
    }
    ws[warp][lane] = warp_sum32d(lo);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        for (int o = 16; o > 0; o >>= 1) hi[i] += __shfl_xor_sync(0xffffffffu, hi[i], o);
        if (lane == 0) ws[warp][32 + i] = hi[i];
    }
    const unsigned total = __reduce_add_sync(0xffffffffu, (unsigned)count);
    if (lane == 0) ws[warp][35] = (double)total;
    __syncthreads();
    if (threadIdx.x < kEpiSums) {
        double t = 0.0;
        for (int w = 0; w < kEpiAccWarps; ++w) t += ws[w][threadIdx.x];
        e.partial[(size_t)blockIdx.x * kEpiSums + threadIdx.x] = t;
    }
}

// The partials are summed in a fixed order, eight threads a sum. The eigenvector of
// the smallest eigenvalue of the 9 x 9 A^T A is taken by inverse iteration started at
// the winning sample's E, with the inverse of A^T A + d I (d = 1e-13 trace: the shift
// keeps the eigenvectors and makes an exactly singular A^T A, as from noiseless
// flows, invertible) from Gauss-Jordan elimination in place, until the iterate moves
// by less than 1e-15 (at most 40 steps; the error shrinks by the ratio of the two
// smallest eigenvalues per step, 0.006 on the driving windows). The result is
// projected again; the four decompositions follow. What bounds it: chains of FP64
// instructions of ~75 cycles each, so the elimination runs on a thread per entry and
// the iteration on a lane per row: 93 us on one thread, now 56 us (the projection is half of it).
constexpr int kEpiSolveParts = 8;

__global__ void __launch_bounds__(kEpiSums * kEpiSolveParts) k_epi_refine_solve(DevParams p, EpiState e)
{
    __shared__ double part[kEpiSolveParts][kEpiSums], sum[kEpiSums], A[9][9], scale[6], xs[9];
    const long long best = e.info[0];
    if (best < 0) return;
    const int tid = threadIdx.x;
    {
        const int i = tid % kEpiSums, c = tid / kEpiSums;
        double t = 0.0;
        for (int b = c; b < e.partial_blocks; b += kEpiSolveParts) t += e.partial[(size_t)b * kEpiSums + i];
        part[c][i] = t;
    }
    if (tid == 0) {
        const double ix = 1.0 / p.fxd, iy = 1.0 / p.fyd;
        scale[0] = ix * ix; scale[1] = ix * iy; scale[2] = ix;
        scale[3] = iy * iy; scale[4] = iy; scale[5] = 1.0;
    }
    __syncthreads();
    if (tid < kEpiSums) {
        double t = 0.0;
        for (int c = 0; c < kEpiSolveParts; ++c) t += part[c][tid];
        sum[tid] = t * (scale[tid / 6] * scale[tid % 6]);
    }
    __syncthreads();
    const double n = sum[kEpiSums - 1];
    // A[(r, c)][(s, d)] = sum of m1_r m1_s m0_c m0_d
    const int row = (tid % 81) / 9, col = tid % 9;
    {
        auto pair = [](int a, int b) { const int lo = min(a, b), hi = max(a, b); return lo == 0 ? hi : lo + hi + 1; };
        if (tid < 81) A[row][col] = sum[pair(row % 3, col % 3) * 6 + pair(row / 3, col / 3)];
    }
    __syncthreads();
    double tr = 0.0;
    for (int i = 0; i < 9; ++i) tr += A[i][i];
    bool ok = n >= 8.0 && tr > 0.0;                        // the same for all threads
    __syncthreads();
    if (tid < 9) A[tid][tid] += 1e-13 * tr;
    __syncthreads();
    for (int k = 0; k < 9 && ok; ++k) {
        const double piv = A[k][k], a = A[row][col], ak = A[row][k], ka = A[k][col];
        ok = piv > 0.0;
        if (!ok) break;
        const double inv = 1.0 / piv;
        const double v = row == k ? (col == k ? inv : ka * inv) : (col == k ? -(ak * inv) : a - ak * (ka * inv));
        __syncthreads();
        if (tid < 81) A[row][col] = v;
        __syncthreads();
    }
    if (tid >= 32) return;
    if (ok) {
        const int i = min(tid, 8);
        double B[9], x = tid < 9 ? e.E[best * 9 + tid] : 0.0;
#pragma unroll
        for (int k = 0; k < 9; ++k) B[k] = A[i][k];
        for (int it = 0; it < 40; ++it) {
            double z[3] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int k = 0; k < 9; ++k) z[k % 3] += B[k] * __shfl_sync(0xffffffffu, x, k);
            const double y = tid < 9 ? (z[0] + z[1]) + z[2] : 0.0;
            double nz = y * y;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) nz += __shfl_xor_sync(0xffffffffu, nz, o);
            const double zi = y * (1.0 / sqrt(nz));
            double step = (zi - x) * (zi - x);
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) step += __shfl_xor_sync(0xffffffffu, step, o);
            x = zi;
            if (__shfl_sync(0xffffffffu, step, 0) < 1e-30) break;
        }
        if (tid < 9) xs[tid] = x;
    }
    __syncwarp();
    if (tid != 0) return;
    e.info[3] = (long long)n;
    double E[9], U[9], Vv[9];
    if (ok) {
        double x[9];
        for (int i = 0; i < 9; ++i) x[i] = xs[i];
        ok = essential_project(x, E, U, Vv);
    }
    if (!ok)
        for (int i = 0; i < 9; ++i) {
            E[i] = e.E[best * 9 + i];
            U[i] = e.UV[best * 18 + i];
            Vv[i] = e.UV[best * 18 + 9 + i];
        }
    for (int i = 0; i < 9; ++i) { e.refined[i] = E[i]; e.refined[9 + i] = U[i]; e.refined[18 + i] = Vv[i]; }
    for (int a = 0; a < 2; ++a) {
        double R[9];
        rot_candidate(U, Vv, a, R);
        for (int sg = 0; sg < 2; ++sg) {
            double* o = e.cand + (2 * a + sg) * 12;
            for (int r = 0; r < 3; ++r) {
                for (int c = 0; c < 3; ++c) o[r * 4 + c] = R[r * 3 + c];
                o[r * 4 + 3] = (sg == 0 ? 1.0 : -1.0) * U[r * 3 + 2];
            }
        }
    }
}

// ---------------------------------------------------------------------------
// 5. Cheirality and T_1
// ---------------------------------------------------------------------------
// The pixel's count for each candidate in FP64 (the definition).
__device__ __noinline__ unsigned cheirality64(const DevParams& p, float2 f, int x, int y, const double* Cd)
{
    unsigned in = 0;
    const double m0x = ((double)x - p.cxd) / p.fxd, m0y = ((double)y - p.cyd) / p.fyd;
    const double m1x = ((double)x + (double)f.x - p.cxd) / p.fxd, m1y = ((double)y + (double)f.y - p.cyd) / p.fyd;
    for (int i = 0; i < 4; ++i) {
        const double* T = Cd + 12 * i;
        const double Rx = T[0] * m0x + T[1] * m0y + T[2];
        const double Ry = T[4] * m0x + T[5] * m0y + T[6];
        const double Rz = T[8] * m0x + T[9] * m0y + T[10];
        const double ax = Rx - m1x * Rz, bx = m1x * T[11] - T[3];
        const double ay = Ry - m1y * Rz, by = m1y * T[11] - T[7];
        const double aa = ax * ax + ay * ay, ab = ax * bx + ay * by;
        if (!(aa > 0.0) || !(ab > 0.0)) continue;
        const double z1 = (ab / aa) * Rz + T[11];
        if (z1 > 0.0) in |= 1u << i;
    }
    return in;
}

// Only the signs of ab and of ab Rz + aa t_z count, so they are taken in FP32 from
// the records, each beside a bound of its error, and a pixel one of whose signs the
// bound leaves open goes to FP64. With u = 2^-24, |R m0| <= n = 1 + |m0x| + |m0y|
// and m = |m0| + |d| (largest component), |t| = 1: a is known to 8 u n (1 + m), b to
// 8 u (1 + m), Rz to 8 u n, and the rest is products; the bounds are taken twice.
// All in FP64 this took 117 us at 1242 x 375; now 14.6 us.
// The last block to finish takes the candidate with the largest count.
__global__ void __launch_bounds__(kEpiThreads) k_epi_cheirality(DevParams p, DevState s, EpiState e, double baseline)
{
    __shared__ double Cd[48];
    __shared__ float Cf[48];
    __shared__ unsigned total[4];
    if (e.info[0] < 0) return;
    if (threadIdx.x < 48) {
        Cd[threadIdx.x] = e.cand[threadIdx.x];
        Cf[threadIdx.x] = (float)e.cand[threadIdx.x];
    }
    if (threadIdx.x < 4) total[threadIdx.x] = 0;
    __syncthreads();
    unsigned cnt[4] = {0, 0, 0, 0};
    constexpr float kU = 0x1p-24f;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < p.N; j += gridDim.x * blockDim.x) {
        const float4 r = e.rec[j];
        if (r.x != r.x) continue;
        const float m0x = r.x, m0y = r.y, m1x = r.x + r.z, m1y = r.y + r.w;
        const float n = 1.f + fabsf(m0x) + fabsf(m0y);
        const float m = 1.f + fmaxf(fabsf(m0x) + fabsf(r.z), fabsf(m0y) + fabsf(r.w));
        const float eb = 16.f * kU * m, ea = eb * n, er = 16.f * kU * n;
        unsigned in = 0;
        bool open = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float* T = Cf + 12 * i;
            const float Rx = fmaf(T[0], m0x, fmaf(T[1], m0y, T[2]));
            const float Ry = fmaf(T[4], m0x, fmaf(T[5], m0y, T[6]));
            const float Rz = fmaf(T[8], m0x, fmaf(T[9], m0y, T[10]));
            const float ax = fmaf(-m1x, Rz, Rx), bx = fmaf(m1x, T[11], -T[3]);
            const float ay = fmaf(-m1y, Rz, Ry), by = fmaf(m1y, T[11], -T[7]);
            const float aa = fmaf(ax, ax, ay * ay), ab = fmaf(ax, bx, ay * by);
            const float sa = fabsf(ax) + fabsf(ay), sb = fabsf(bx) + fabsf(by);
            const float e_ab = fmaf(2.f * eb, sa, ea * (sb + 2.f * eb));
            const float e_aa = 2.f * ea * (sa + ea) + 8.f * kU * aa;
            const float z = fmaf(ab, Rz, aa * T[11]);
            const float e_z = e_ab * n + fabsf(ab) * er + e_aa + 8.f * kU * (fabsf(ab) * n + aa);
            if (ab < -e_ab) continue;
            if (!(ab > e_ab && fabsf(z) > e_z)) open = true;
            else if (z > 0.f) in |= 1u << i;
        }
        if (open) in = cheirality64(p, load_flow(s.flows, p.flow_f16, (size_t)j), j % p.W, j / p.W, Cd);
#pragma unroll
        for (int i = 0; i < 4; ++i) cnt[i] += (in >> i) & 1u;
    }
    for (int i = 0; i < 4; ++i) {
        const unsigned v = __reduce_add_sync(0xffffffffu, cnt[i]);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&total[i], v);
    }
    __syncthreads();
    if (threadIdx.x < 4 && total[threadIdx.x])
        atomicAdd((unsigned long long*)(e.info + 4 + threadIdx.x), (unsigned long long)total[threadIdx.x]);
    __syncthreads();
    if (threadIdx.x != 0) return;
    __threadfence();
    if (atomicAdd(e.cheirality_done, 1) != (int)gridDim.x - 1) return;
    __threadfence();
    int c = 0;
    for (int i = 1; i < 4; ++i)
        if (__ldcg(e.info + 4 + i) > __ldcg(e.info + 4 + c)) c = i;
    e.info[1] = c;
    for (int r = 0; r < 3; ++r) {
        for (int q = 0; q < 3; ++q) e.T1[r * 4 + q] = Cd[12 * c + r * 4 + q];
        e.T1[r * 4 + 3] = baseline * Cd[12 * c + r * 4 + 3];
    }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
constexpr int kEpiCheiralityBlocks = 2 * 152;

// Collected errors a sample has room for: a sixteenth of the pixels (the bracket
// holds a few percent), within these bounds.
constexpr int kEpiCapMin = 4096, kEpiCapMax = 65536;

// Carves the scratch for M samples out of `base` (which may be null to measure)
// and returns the bytes it spans; every piece starts on a 256-byte boundary.
size_t epi_layout(void* base, int M, int W, int H, float4* rec, EpiState* e)
{
    const int N = W * H;
    const uintptr_t start = reinterpret_cast<uintptr_t>(base);
    size_t off = 0;
    auto take = [&](size_t n) {
        void* r = reinterpret_cast<void*>(start + off);
        off += (n + 255) & ~(size_t)255;
        return r;
    };
    e->M = M;
    e->rec = rec;
    e->valid = static_cast<int*>(take((size_t)M * 4));
    e->E = static_cast<double*>(take((size_t)M * 9 * 8));
    e->UV = static_cast<double*>(take((size_t)M * 18 * 8));
    e->form = static_cast<float*>(take((size_t)M * 12 * 4));
    e->list = static_cast<int*>(take((size_t)M * 4));
    e->lo = static_cast<unsigned*>(take((size_t)M * 4));
    e->hi = static_cast<unsigned*>(take((size_t)M * 4));
    e->cap = N / 16 < kEpiCapMin ? kEpiCapMin : (N / 16 > kEpiCapMax ? kEpiCapMax : N / 16);
    e->found = static_cast<unsigned*>(take((size_t)M * e->cap * 4));
    // zeroed together before every estimate: zero .. zero + zero_bytes
    const size_t z0 = off;
    e->zero = reinterpret_cast<void*>(start + off);
    e->below = static_cast<unsigned*>(take((size_t)M * 4));
    e->inside = static_cast<unsigned*>(take((size_t)M * 4));
    e->n_list = static_cast<int*>(take(4));
    e->done = static_cast<int*>(take(4));
    e->median_done = static_cast<int*>(take(4));
    e->cheirality_done = static_cast<int*>(take(4));
    e->info = static_cast<long long*>(take(8 * 8));
    e->zero_bytes = off - z0;
    e->median = static_cast<float*>(take((size_t)M * 4));
    e->partial_blocks = (((W + 31) / 32) * ((H + kEpiAccRows - 1) / kEpiAccRows) + kEpiAccWarps - 1) / kEpiAccWarps;
    e->partial = static_cast<double*>(take((size_t)e->partial_blocks * kEpiSums * 8));
    e->refined = static_cast<double*>(take(27 * 8));
    e->cand = static_cast<double*>(take(48 * 8));
    e->T1 = static_cast<double*>(take(12 * 8));
    return off;
}

size_t epi_scratch_bytes(int M, int W, int H)
{
    EpiState e;
    return epi_layout(nullptr, M, W, H, nullptr, &e);
}

// Enqueues the whole estimate on st; returns the number of kernels launched.
int launch_epipolar(const DevParams& p, const DevState& s, const EpiState& e, double baseline, cudaStream_t st)
{
    int k = 0;
    cudaMemsetAsync(e.zero, 0, e.zero_bytes, st);
    k_epi_records<<<dim3((p.W + 31) / 32, (p.H + kEpiRecRows * kEpiRecWarps - 1) / (kEpiRecRows * kEpiRecWarps)),
                    32 * kEpiRecWarps, 0, st>>>(p, s, e); ++k;
    k_epi_samples<<<(e.M * kEpiSampleLanes + kEpiSampleBlock - 1) / kEpiSampleBlock, kEpiSampleBlock, 0, st>>>(p, s, e); ++k;
    k_epi_bracket<<<e.M, kEpiSubThreads, 0, st>>>(p, e); ++k;
    // persistent blocks: the number of valid samples is known on the device only
    k_epi_count<<<3 * 152, kEpiThreads, 0, st>>>(p, e); ++k;
    k_epi_median<<<e.M, kEpiMedianThreads, 0, st>>>(p, e); ++k;
    k_epi_refine_accum<<<e.partial_blocks, 32 * kEpiAccWarps, 0, st>>>(p, s, e); ++k;
    k_epi_refine_solve<<<1, kEpiSums * kEpiSolveParts, 0, st>>>(p, e); ++k;
    k_epi_cheirality<<<kEpiCheiralityBlocks, kEpiThreads, 0, st>>>(p, s, e, baseline); ++k;
    return k;
}

}  // namespace vd
