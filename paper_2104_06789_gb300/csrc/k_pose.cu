// Pose-update kernels (Sec. 5.2): Monte-Carlo minimal groups drawn with
// Philox4x64-10, FP64 P3P per group (Eq. 17), order-preserving hypothesis
// collection with se(3) logarithms, and the weighted Gaussian meanshift of
// Eqs. 18-19 on a thread-block cluster.
#include <algorithm>

#include <cooperative_groups.h>

#include "df32.cuh"
#include "score_ops.cuh"
#include "voldor_internal.cuh"

namespace cg = cooperative_groups;

namespace vd {

// ---------------------------------------------------------------------------
// FP64 helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ double d3dot(const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

__device__ __forceinline__ void d3cross(const double* a, const double* b, double* o)
{
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ bool d3unit(double* a)
{
    const double n = sqrt(d3dot(a, a));
    if (!(n > 0.0)) return false;
    const double r = 1.0 / n;
    a[0] *= r; a[1] *= r; a[2] *= r;
    return true;
}

__device__ __forceinline__ double horner4(const double* c, double x)
{
    return (((c[4] * x + c[3]) * x + c[2]) * x + c[1]) * x + c[0];
}

// a / b, correctly rounded, from y = 1 / b correctly rounded, for quotients and
// remainders inside the normal range: the first correction brings q within one ulp,
// and the second then rounds correctly (Markstein, IBM J. Res. Dev. 34, 1990). Five
// FP64 instructions where the division takes about twelve.
__device__ __forceinline__ double div_by(double a, double b, double y)
{
    double q = a * y;
    q = fma(fma(-b, q, a), y, q);
    return fma(fma(-b, q, a), y, q);
}

__device__ __forceinline__ double third(double a) { return div_by(a, 3.0, 1.0 / 3.0); }

// Largest real root of m^3 + A m^2 + B m + C (Cardano or trigonometric form),
// refined by Newton steps; all lanes of the quad on the same coefficients, the two
// cube roots on its even and odd lanes. Every lane of the warp takes part.
__device__ double cubic_max_root(double A, double B, double C)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, base = lane & ~3;
    const double A3 = third(A);
    const double pp = B - A * A3;                         // y^3 + pp y + qq = 0, m = y - A/3
    const double qq = 2.0 * A3 * A3 * A3 - A3 * B + C;
    const double disc = 0.25 * qq * qq + div_by(pp * pp * pp, 27.0, 1.0 / 27.0);
    const bool one = disc > 0.0;
    double part = 0.0;
    if (one) {
        const double sq = sqrt(disc);
        part = cbrt(-0.5 * qq + (lane & 1 ? -sq : sq));
    }
    double y = __shfl_sync(FULL, part, base) + __shfl_sync(FULL, part, base + 1);
    if (!one) {
        const double r = sqrt(fmax(third(-pp), 0.0));
        double arg = (r > 0.0) ? (-0.5 * qq) / (r * r * r) : 0.0;
        arg = fmin(1.0, fmax(-1.0, arg));
        y = 2.0 * r * cos(third(acos(arg)));
    }
    double m = y - A3;
    double f = ((m + A) * m + B) * m + C;
    for (int it = 0; it < 4; ++it) {
        const double df = (3.0 * m + 2.0 * A) * m + B;
        if (!(fabs(df) > 0.0)) break;
        const double mn = m - f / df;
        const double fn = ((mn + A) * mn + B) * mn + C;
        if (!(fabs(fn) < fabs(f))) break;
        m = mn;
        f = fn;
    }
    return m;
}

// Lane r's root candidate of a quartic (ascending coefficients, the same in all lanes
// of a quad) by Ferrari's method, before polishing, shifted back by -b/4; false if it
// has none. The quad's candidates, in lane order: the two roots of the first
// quadratic factor, then those of the second. Every lane of the warp takes part.
__device__ bool quartic_candidate(const double* a, double& root)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, r = lane & 3, base = lane & ~3;
    double amax = 0.0;
    for (int i = 0; i < 4; ++i) amax = fmax(amax, fabs(a[i]));
    const double own = (r == 0 ? a[3] : (r == 1 ? a[2] : (r == 2 ? a[1] : a[0]))) / a[4];
    const double b = __shfl_sync(FULL, own, base), c = __shfl_sync(FULL, own, base + 1);
    const double d = __shfl_sync(FULL, own, base + 2), e = __shfl_sync(FULL, own, base + 3);
    const double bb = b * b;
    const double P = c - 0.375 * bb;
    const double Q = d - 0.5 * b * c + 0.125 * bb * b;
    const double R = e - 0.25 * b * d + 0.0625 * bb * c - (3.0 / 256.0) * bb * bb;
    // y^4 + P y^2 + Q y + R = (y^2 + P/2 + m)^2 - 2m (y - Q/(4m))^2 for the
    // resolvent root m of m^3 + P m^2 + (P^2/4 - R) m - Q^2/8 = 0
    const double m = cubic_max_root(P, 0.25 * P * P - R, -0.125 * Q * Q);
    if (!(fabs(a[4]) > 1e-14 * amax)) return false;       // degenerate group
    double y;
    if (m > 1e-300 && fabs(Q) > 0.0) {
        const double sr = sqrt(2.0 * m);
        const double h = Q / (2.0 * sr);
        const double cf = 0.5 * P + m + (r < 2 ? -h : h), D = 2.0 * m - 4.0 * cf;
        if (!(D >= 0.0)) return false;
        const double q = sqrt(D);
        y = 0.5 * ((r < 2 ? -sr : sr) + (r & 1 ? -q : q));
    } else {
        const double D = P * P - 4.0 * R;                 // biquadratic y^4 + P y^2 + R
        if (!(D >= 0.0)) return false;
        const double sq = sqrt(D), z = 0.5 * (-P + (r < 2 ? sq : -sq));
        if (!(z >= 0.0)) return false;
        y = sqrt(z);
        if (r & 1) y = -y;
    }
    root = y - 0.25 * b;
    return true;
}

// One candidate root polished by Newton steps on the quartic.
__device__ double polish_quartic_root(const double* a, double x)
{
    double f = horner4(a, x);
    for (int it = 0; it < 3; ++it) {
        const double df = ((4.0 * a[4] * x + 3.0 * a[3]) * x + 2.0 * a[2]) * x + a[1];
        if (!(fabs(df) > 0.0)) break;
        const double xn = x - f / df, fn = horner4(a, xn);
        if (!(fabs(fn) < fabs(f))) break;
        x = xn;
        f = fn;
    }
    return x;
}

// Frame spanned by a triangle: f1 along q3 - q1, f3 normal, f2 = f3 x f1
// (columns of F, row-major).
__device__ __forceinline__ bool tri_frame(const double* q1, const double* q2, const double* q3, double* F)
{
    double f1[3] = {q3[0] - q1[0], q3[1] - q1[1], q3[2] - q1[2]};
    const double e[3] = {q2[0] - q1[0], q2[1] - q1[1], q2[2] - q1[2]};
    if (!d3unit(f1)) return false;
    double f3[3];
    d3cross(f1, e, f3);
    if (!d3unit(f3)) return false;
    double f2[3];
    d3cross(f3, f1, f2);
    for (int r = 0; r < 3; ++r) { F[r * 3 + 0] = f1[r]; F[r * 3 + 1] = f2[r]; F[r * 3 + 2] = f3[r]; }
    return true;
}

// ---------------------------------------------------------------------------
// P3P. With s_i the distances along the unit bearings b_i, the law of cosines
// gives s_i^2 + s_k^2 - 2 c_ik s_i s_k = d_ik^2. With u = s2/s1, v = s3/s1:
//   (ii)/(i):  v^2 - 2 c13 v = g(u),  g(u) = (d13/d12)(1 + u^2 - 2 c12 u) - 1
//   with (iii): v D(u) = N(u),  N = d23 (1 + g) - d13 (u^2 + g),
//                               D = 2 d13 (c13 - c23 u)
//   and N^2 - 2 c13 N D - g D^2 = 0 is a quartic in u.
// Each root is polished by Newton steps on the three distance equations; the
// pose maps the world triangle onto the camera triangle. Solutions with all
// s_i > 0 come back sorted by s1.
// ---------------------------------------------------------------------------
struct P3PSol {
    double s1;
    double Rt[12];
};

// The quartic of a P3P instance and the quantities its roots are mapped back
// with. False for a degenerate triangle.
struct P3PSetup {
    double d12, d13, d23, c12, c13, c23;
    double N[3], D[2], Q[5];
};

// Lane r of the quad forms the squared distance and the cosine of points (0, 1),
// (0, 2) or (1, 2) (lane 3 the first again). Every lane of the warp takes part.
__device__ bool p3p_setup(const double P[3][3], const double b[3][3], P3PSetup& q)
{
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, r = lane & 3, base = lane & ~3;
    double e[3], bi[3], bj[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        e[i] = (r == 2 ? P[1][i] : P[0][i]) - (r == 1 || r == 2 ? P[2][i] : P[1][i]);
        bi[i] = r == 2 ? b[1][i] : b[0][i];
        bj[i] = r == 1 || r == 2 ? b[2][i] : b[1][i];
    }
    const double dist = d3dot(e, e), cosine = d3dot(bi, bj);
    const double d12 = __shfl_sync(FULL, dist, base), d13 = __shfl_sync(FULL, dist, base + 1), d23 = __shfl_sync(FULL, dist, base + 2);
    const double c12 = __shfl_sync(FULL, cosine, base), c13 = __shfl_sync(FULL, cosine, base + 1), c23 = __shfl_sync(FULL, cosine, base + 2);
    const double K2 = d13 / d12;
    const double g[3] = {K2 - 1.0, -2.0 * K2 * c12, K2};
    q.d12 = d12; q.d13 = d13; q.d23 = d23; q.c12 = c12; q.c13 = c13; q.c23 = c23;
    q.N[0] = (d23 - d13) * g[0] + d23; q.N[1] = (d23 - d13) * g[1]; q.N[2] = (d23 - d13) * g[2] - d13;
    q.D[0] = 2.0 * d13 * c13; q.D[1] = -2.0 * d13 * c23;
    const double* N = q.N;
    const double* D = q.D;
    for (int i = 0; i < 5; ++i) q.Q[i] = 0.0;
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) q.Q[i + j] += N[i] * N[j];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 2; ++j) q.Q[i + j] -= 2.0 * c13 * N[i] * D[j];
    const double DD[3] = {D[0] * D[0], 2.0 * D[0] * D[1], D[1] * D[1]};
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j) q.Q[i + j] -= g[i] * DD[j];
    return d12 > 0.0 && d13 > 0.0 && d23 > 0.0;
}

// The pose of one polished root u of the quartic: v, the distances s_i
// (polished by Newton steps on the three distance equations), then the
// rotation and translation that map the world triangle onto the camera
// triangle. False if the root gives no solution with all s_i > 0.
__device__ bool p3p_from_root(const double P[3][3], const double b[3][3], const P3PSetup& q, const double u,
                              P3PSol& sol)
{
    const double d12 = q.d12, d13 = q.d13, d23 = q.d23, c12 = q.c12, c13 = q.c13, c23 = q.c23;
    const double* N = q.N;
    const double* D = q.D;
    if (!(u > 0.0)) return false;
    const double Du = D[0] + D[1] * u;
    if (Du == 0.0) return false;
    const double v = (N[0] + (N[1] + N[2] * u) * u) / Du;
    const double q1 = 1.0 + u * u - 2.0 * c12 * u;
    if (!(q1 > 0.0)) return false;
    double s[3];
    s[0] = sqrt(d12 / q1);
    s[1] = u * s[0];
    s[2] = v * s[0];
    if (!(s[0] > 0.0 && s[1] > 0.0 && s[2] > 0.0) || !isfinite(s[2])) return false;
    // residuals of the three equations; J = 2 {j0 j1 0; j2 0 j3; 0 j4 j5} is solved
    // through the adjugate of the half, whose entries are single products
    auto residuals = [&](const double* s, double* F) {
        F[0] = s[0] * s[0] + s[1] * s[1] - 2.0 * c12 * s[0] * s[1] - d12;
        F[1] = s[0] * s[0] + s[2] * s[2] - 2.0 * c13 * s[0] * s[2] - d13;
        F[2] = s[1] * s[1] + s[2] * s[2] - 2.0 * c23 * s[1] * s[2] - d23;
    };
    double F[3];
    residuals(s, F);
    for (int it = 0; it < 5; ++it) {
        const double j0 = s[0] - c12 * s[1], j1 = s[1] - c12 * s[0], j2 = s[0] - c13 * s[2], j3 = s[2] - c13 * s[0],
                     j4 = s[1] - c23 * s[2], j5 = s[2] - c23 * s[1];
        const double c00 = -(j3 * j4), c01 = -(j2 * j5), c02 = j2 * j4, c10 = -(j1 * j5), c11 = j0 * j5, c12_ = -(j0 * j4),
                     c20 = j1 * j3, c21 = -(j0 * j3), c22 = -(j1 * j2);
        const double det = j0 * c00 + j1 * c01;
        if (!(fabs(det) > 0.0)) break;
        const double id = 0.5 * (1.0 / det);
        const double ns[3] = {s[0] - (c00 * F[0] + c10 * F[1] + c20 * F[2]) * id, s[1] - (c01 * F[0] + c11 * F[1] + c21 * F[2]) * id,
                              s[2] - (c02 * F[0] + c12_ * F[1] + c22 * F[2]) * id};
        double G[3];
        residuals(ns, G);
        if (!(fabs(G[0]) + fabs(G[1]) + fabs(G[2]) < fabs(F[0]) + fabs(F[1]) + fabs(F[2]))) break;
        for (int i = 0; i < 3; ++i) { s[i] = ns[i]; F[i] = G[i]; }
    }
    if (!(s[0] > 0.0 && s[1] > 0.0 && s[2] > 0.0)) return false;
    double Qc[3][3];
    for (int i = 0; i < 3; ++i)
        for (int c = 0; c < 3; ++c) Qc[i][c] = s[i] * b[i][c];
    double Fw[9], Fc[9];
    if (!tri_frame(P[0], P[1], P[2], Fw) || !tri_frame(Qc[0], Qc[1], Qc[2], Fc)) return false;
    sol.s1 = s[0];
    double cw[3], cc[3];
    for (int c = 0; c < 3; ++c) {
        cw[c] = third(P[0][c] + P[1][c] + P[2][c]);
        cc[c] = third(Qc[0][c] + Qc[1][c] + Qc[2][c]);
    }
    for (int r0 = 0; r0 < 3; ++r0) {
        for (int c = 0; c < 3; ++c)
            sol.Rt[r0 * 4 + c] = Fc[r0 * 3 + 0] * Fw[c * 3 + 0] + Fc[r0 * 3 + 1] * Fw[c * 3 + 1] + Fc[r0 * 3 + 2] * Fw[c * 3 + 2];
    }
    for (int r0 = 0; r0 < 3; ++r0)
        sol.Rt[r0 * 4 + 3] = cc[r0] - (sol.Rt[r0 * 4 + 0] * cw[0] + sol.Rt[r0 * 4 + 1] * cw[1] + sol.Rt[r0 * 4 + 2] * cw[2]);
    return true;
}

// ---------------------------------------------------------------------------
// Minimal groups of frame t at iteration k (Sec. 5.2): the pixels with a 3D-2D
// correspondence (pi_{t-1} valid), in pixel order, form the list V_t of n
// entries; Philox(index g, t, k, POSE) gives j_i = V_t[hi64(r_i * n)] and a
// group with a repeated pixel yields nothing. P3P (Eq. 17) takes the points in
// camera t-1 and the bearings of the flow targets pi_{t-1} + X_t in camera t,
// all in FP64.
// ---------------------------------------------------------------------------

// The i-th valid pixel of the frame (0 <= i < n): the block whose record
// offset is the last one <= i (the count pass's exclusive scan), then the
// (i - offset)-th set bit of that block's per-warp ballots.
__device__ int valid_pixel_at(const DevState& s, int nb, int i)
{
    // the last of the nb offsets that is <= i: seven probes a round, all in flight
    int lo = 0, n = nb;
    while (n > 1) {
        const int step = (n + 7) >> 3;
        int below = 0;
#pragma unroll
        for (int q = 1; q < 8; ++q) {
            const int at = q * step;
            below += at < n && s.pix_block_count[lo + at] <= i;
        }
        lo += below * step;
        n = min(step, n - below * step);
    }
    int r = i - s.pix_block_count[lo];
    const uint4* m4 = reinterpret_cast<const uint4*>(s.pix_vmask + (size_t)lo * (kPixThreads / 32));
    static_assert(kPixThreads == 256, "eight ballots a block");
    const uint4 ma = m4[0], mb = m4[1];
    const unsigned m[8] = {ma.x, ma.y, ma.z, ma.w, mb.x, mb.y, mb.z, mb.w};
#pragma unroll
    for (int w = 0; w < kPixThreads / 32; ++w) {
        const int c = __popc(m[w]);
        if (r < c) {                                      // its r-th set bit
            unsigned mw = m[w];
            int bit = 0;
#pragma unroll
            for (int h = 16; h > 0; h >>= 1) {
                const int low = __popc(mw & ((1u << h) - 1u));
                if (r >= low) { r -= low; mw >>= h; bit += h; }
            }
            return lo * kPixThreads + w * 32 + bit;
        }
        r -= c;
    }
    return -1;
}

// a / f for a focal length f with y = 1 / f rounded.
__device__ __forceinline__ double by_focal(double a, double f, double y)
{
    return f > 1e-60 && f < 1e60 && fabs(a) < 1e60 ? div_by(a, f, y) : a / f;
}

// Point in camera t-1 and bearing of the flow target of valid pixel j, in
// FP64 (P3P's inputs): P = C_{t-1} theta K^-1 [x y 1], pi_{t-1} its
// projection (the pixel itself for t = 1), the flow X_t sampled bilinearly at
// pi_{t-1}. False if the pixel has no correspondence after all (the pose
// preparation lists it by the same test in float-float; the two can differ
// only within ~1e-11 px of the image border).
__device__ bool group_point(const DevParams& p, const DevState& s, const double* C, int t, int j, double* P,
                            double* bear)
{
    const int x = j % p.W, y = j / p.W;
    const double th = (double)s.theta[j];
    const double d[3] = {by_focal((double)x - p.cxd, p.fxd, p.inv_fxd), by_focal((double)y - p.cyd, p.fyd, p.inv_fyd), 1.0};
    double u, v;
    if (t == 1) {
        P[0] = th * d[0]; P[1] = th * d[1]; P[2] = th;
        u = x; v = y;
        if (!(P[2] > 0.0)) return false;
    } else {
        const double X = th * d[0], Y = th * d[1], Z = th;
        for (int r = 0; r < 3; ++r) P[r] = C[r * 4 + 0] * X + C[r * 4 + 1] * Y + C[r * 4 + 2] * Z + C[r * 4 + 3];
        if (!(P[2] > 0.0)) return false;
        u = p.fxd * P[0] / P[2] + p.cxd;
        v = p.fyd * P[1] / P[2] + p.cyd;
    }
    if (!(u >= 0.0 && u <= (double)(p.W - 1) && v >= 0.0 && v <= (double)(p.H - 1))) return false;
    const int x0 = min((int)floor(u), p.W - 2), y0 = min((int)floor(v), p.H - 2);
    const double ax = u - x0, ay = v - y0;
    const size_t base = (size_t)(t - 1) * p.N + (size_t)y0 * p.W + x0;
    const float2 f00 = load_flow(s.flows, p.flow_f16, base), f10 = load_flow(s.flows, p.flow_f16, base + 1);
    const float2 f01 = load_flow(s.flows, p.flow_f16, base + p.W), f11 = load_flow(s.flows, p.flow_f16, base + p.W + 1);
    const double w00 = (1 - ax) * (1 - ay), w10 = ax * (1 - ay), w01 = (1 - ax) * ay, w11 = ax * ay;
    const double fu = w00 * f00.x + w10 * f10.x + w01 * f01.x + w11 * f11.x;
    const double fv = w00 * f00.y + w10 * f10.y + w01 * f01.y + w11 * f11.y;
    bear[0] = by_focal(u + fu - p.cxd, p.fxd, p.inv_fxd);
    bear[1] = by_focal(v + fv - p.cyd, p.fyd, p.inv_fyd);
    bear[2] = 1.0;
    return d3unit(bear);
}

// Groups are solved in order in chunks of kP3PChunk (one warp each: four
// lanes per group, one per root of its quartic) until the frame has S
// solutions or the budget of G groups is spent. A warp claims chunks with an
// atomic counter, so the claimed chunks are always 0, 1, ..., c - 1, and every
// claimed chunk is solved: the solved groups form a prefix of the group order.
// After its first chunk a warp claims another only while the solutions found
// so far plus the chunks still in flight, at the yield observed so far, fall
// short of S; the warp that completes the last chunk in flight sees exact
// counts, so the run ends with at least S solutions in the prefix (or the
// whole budget solved), and the first S solutions in group order are the same
// whatever the timing.
//
// Within a quad, lanes 0-2 compute the FP64 point and bearing of the group's
// pixels 0-2 and share them by shuffles; the lanes share the work on the quartic (the
// pairs of points, its division by the leading coefficient, the cube roots), lane r
// forms and polishes root candidate r and turns it into a pose, and each solution's
// slot is its rank by s1 among the quad's solutions (ties by root order): the group's
// solutions sorted by s1. A warp's FP64 work is then the common part and one root,
// not up to four roots in turn.
//
// What bounds it is the number of FP64 instructions of a warp: one issues every ~54
// cycles from a single warp whether or not it depends on the last, and an SM takes
// three and a half such warps before they slow each other down. So nothing is
// computed in two lanes that one can do, divisions by constants go through their
// reciprocals, a Newton step keeps its residual for the next and leaves out the zeros
// of its matrix: 53 -> 45 us up to S = 2048, 58 -> 50 at 4096, 77 -> 64 at 8192.
__global__ void __launch_bounds__(32) k_p3p_groups(DevParams p, DevState s, int t)
{
    const int lane = threadIdx.x, quad = lane >> 2, r = lane & 3, base = lane & ~3;
    const unsigned FULL = 0xffffffffu;
    const int n_valid = *s.pix_count;
    if (n_valid < 3) return;                              // every group repeats a pixel
    const int k = *s.iter;
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    const int n_chunks = (p.G + kP3PChunk - 1) / kP3PChunk;
    const double* C = s.cum + 12 * (t - 1);
    bool first = true;
    for (;;) {
        int c = -1;
        if (lane == 0) {
            bool claim = first;
            if (!first) {
                const unsigned long long d = atomicAdd(s.p3p_done, 0ull);
                const long long done = (long long)(d >> 32), sols = (long long)(d & 0xffffffffull);
                const long long inflight = max(0LL, (long long)atomicAdd(s.p3p_claims, 0) - done);
                claim = sols + (done > 0 ? inflight * sols / done : inflight) < (long long)p.S;
            }
            if (claim) c = atomicAdd(s.p3p_claims, 1);
        }
        first = false;
        c = __shfl_sync(FULL, c, 0);
        if (c < 0 || c >= n_chunks) break;
        const int g = c * kP3PChunk + quad;
        const bool active = g < p.G;
        // the group's pixels: j_i = V_t[hi64(r_i n)] (all lanes of the quad draw the same)
        int idx[3] = {0, 0, 0};
        bool distinct = false;
        if (active) {
            const U64x4 rr = philox4x64_10((uint64_t)g, (uint64_t)t, (uint64_t)k, (uint64_t)kStreamPose, p.seed,
                                           p.window_id);
            for (int i = 0; i < 3; ++i) idx[i] = (int)__umul64hi(rr.v[i], (uint64_t)n_valid);
            distinct = idx[0] != idx[1] && idx[0] != idx[2] && idx[1] != idx[2];
        }
        // lane r < 3: pixel r's point in camera t-1 and bearing (FP64)
        double Pm[3] = {0.0, 0.0, 0.0}, bm[3] = {0.0, 0.0, 1.0};
        double wv = 0.0;
        int ok = 1;
        if (active && distinct && r < 3) {
            const int ri = r == 0 ? idx[0] : (r == 1 ? idx[1] : idx[2]);
            const int j = valid_pixel_at(s, nb, ri);
            ok = (j >= 0 && group_point(p, s, C, t, j, Pm, bm)) ? 1 : 0;
            if (ok) wv = (double)s.wmap[(size_t)(t - 1) * p.N + j];
        }
        double P[3][3], b[3][3];
        double weight = 1.0;
        int okall = 1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                P[i][q] = __shfl_sync(FULL, Pm[q], base + i);
                b[i][q] = __shfl_sync(FULL, bm[q], base + i);
            }
            weight *= __shfl_sync(FULL, wv, base + i);
            okall &= __shfl_sync(FULL, ok, base + i);
        }
        const bool valid_group = active && distinct && okall;
        if (!valid_group) weight = 0.0;
        // the quartic (every lane), then lane r's root
        P3PSetup qs;
        double u0 = 0.0;
        const bool set = p3p_setup(P, b, qs), some = quartic_candidate(qs.Q, u0);
        P3PSol sol;
        sol.s1 = 0.0;
        bool has = false;
        if (valid_group && set && some) {
            has = p3p_from_root(P, b, qs, polish_quartic_root(qs.Q, u0), sol);
        }
        // slot = rank by s1 among the quad's solutions, ties by root order
        int rank = 0, cnt = 0;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
            const double so = __shfl_sync(FULL, sol.s1, base + o);
            const int ho = __shfl_sync(FULL, has ? 1 : 0, base + o);
            cnt += ho;
            if (has && ho && (so < sol.s1 || (so == sol.s1 && o < r))) ++rank;
        }
        if (active) {
            if (r == 0) {
                s.grp_count[g] = cnt;
                s.grp_weight[g] = weight;
            }
            if (has) {
                double* o = s.grp_sols + ((size_t)g * kMaxSols + rank) * 12;
                for (int q = 0; q < 12; ++q) o[q] = sol.Rt[q];
            }
        }
        int tot = (r == 0) ? cnt : 0;
        for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(FULL, tot, o);
        __threadfence();
        if (lane == 0) {
            s.chunk_sols[c] = tot;
            if (tot) atomicAdd(s.block_sols + c / kP3PBlock, tot);
            atomicAdd(s.p3p_done, (1ull << 32) | (unsigned long long)tot);
        }
    }
}

// Groups solved for the current frame (a prefix of the group order).
__device__ __forceinline__ int groups_solved(const DevParams& p, const DevState& s)
{
    const int n_chunks = (p.G + kP3PChunk - 1) / kP3PChunk;
    return min(min(*s.p3p_claims, n_chunks) * kP3PChunk, p.G);
}

// One warp per block spreads the FP64 solves over the SMs. The first wave takes S
// groups (more than one solution each as a rule), so that no warp runs a second chunk
// after its first, a whole chain later: with 3/4 S groups, enough only above 1.33
// solutions a group, frames of handheld windows take 64 us on average (46 or 81) at
// S = 4096 on 640 x 480 where S groups take 48, and 68 against 45 at S = 2048 on
// 320 x 240. An SM solves three and a half chunks in the time of one and no more (5/4 S
// groups at S = 4096: 57 us), so beyond kP3PFreeChunks chunks in all it is 3/4 S, as the
// yield of driving windows (1.4-1.5) allows (S = 8192: 64 us; with S groups 73, with 5/4 S
// 93); further chunks are claimed as needed.
constexpr int kP3PFreeChunks = 512;

void launch_p3p_groups(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    const int n_chunks = (p.G + kP3PChunk - 1) / kP3PChunk;
    const int all = (p.S + kP3PChunk - 1) / kP3PChunk, most = (3 * p.S + 4 * kP3PChunk - 1) / (4 * kP3PChunk);
    const int wave = std::min(n_chunks, std::max(most, std::min(all, kP3PFreeChunks)));
    k_p3p_groups<<<wave, 32, 0, st>>>(p, s, t);
}

// se(3) logarithm through the unit quaternion of R (Shepperd's selection):
// phi = 2 atan2(|v|, w) v/|v|, rho = V^-1 t with
// V^-1 = I - Phi/2 + (1 - (th/2) cot(th/2)) / th^2 Phi^2, where
// cot(th/2) = w / |v| (w = cos(th/2), |v| = sin(th/2), w >= 0): no FP64
// sine or cosine, which are long serial routines on this GPU's FP64 pipe.
__device__ void se3_log_quat(const double* Rt, double* p6)
{
    const double R00 = Rt[0], R01 = Rt[1], R02 = Rt[2];
    const double R10 = Rt[4], R11 = Rt[5], R12 = Rt[6];
    const double R20 = Rt[8], R21 = Rt[9], R22 = Rt[10];
    const double tr = R00 + R11 + R22;
    double w, x, y, z;
    if (tr >= R00 && tr >= R11 && tr >= R22) {
        w = 0.5 * sqrt(1.0 + tr);
        const double f = 0.25 / w;
        x = (R21 - R12) * f; y = (R02 - R20) * f; z = (R10 - R01) * f;
    } else if (R00 >= R11 && R00 >= R22) {
        x = 0.5 * sqrt(1.0 + R00 - R11 - R22);
        const double f = 0.25 / x;
        w = (R21 - R12) * f; y = (R01 + R10) * f; z = (R02 + R20) * f;
    } else if (R11 >= R22) {
        y = 0.5 * sqrt(1.0 - R00 + R11 - R22);
        const double f = 0.25 / y;
        w = (R02 - R20) * f; x = (R01 + R10) * f; z = (R12 + R21) * f;
    } else {
        z = 0.5 * sqrt(1.0 - R00 - R11 + R22);
        const double f = 0.25 / z;
        w = (R10 - R01) * f; x = (R02 + R20) * f; y = (R12 + R21) * f;
    }
    if (w < 0.0) { w = -w; x = -x; y = -y; z = -z; }
    const double vn = sqrt(x * x + y * y + z * z);
    const double th = 2.0 * atan2(vn, w);
    const double scale = (vn > 1e-8) ? th / vn : (2.0 / w) * (1.0 - vn * vn / (3.0 * w * w));
    const double phi[3] = {scale * x, scale * y, scale * z};
    double c2;
    if (th < 1e-4) c2 = 1.0 / 12.0 + th * th / 720.0;
    else c2 = (1.0 - 0.5 * th * w / vn) / (th * th);
    const double t[3] = {Rt[3], Rt[7], Rt[11]};
    double a[3], b[3];
    d3cross(phi, t, a);
    d3cross(phi, a, b);
    for (int i = 0; i < 3; ++i) p6[i] = t[i] - 0.5 * a[i] + c2 * b[i];
    p6[3] = phi[0]; p6[4] = phi[1]; p6[5] = phi[2];
}

// se(3) exponential: R = I + A Phi + B Phi^2, t = rho + B phi x rho + C phi x (phi x rho).
__device__ void se3_exp_vec(const double* p6, double* Rt)
{
    const double* rho = p6;
    const double* phi = p6 + 3;
    const double th2 = d3dot(phi, phi), th = sqrt(th2);
    double A, B, C;
    if (th < 1e-4) {
        A = 1.0 - th2 / 6.0 + th2 * th2 / 120.0;
        B = 0.5 - th2 / 24.0 + th2 * th2 / 720.0;
        C = 1.0 / 6.0 - th2 / 120.0 + th2 * th2 / 5040.0;
    } else {
        A = sin(th) / th;
        B = (1.0 - cos(th)) / th2;
        C = (th - sin(th)) / (th2 * th);
    }
    const double wx = phi[0], wy = phi[1], wz = phi[2];
    // Phi^2 = phi phi^T - th^2 I
    Rt[0] = 1.0 + B * (wx * wx - th2); Rt[1] = -A * wz + B * wx * wy;       Rt[2] = A * wy + B * wx * wz;
    Rt[4] = A * wz + B * wx * wy;       Rt[5] = 1.0 + B * (wy * wy - th2); Rt[6] = -A * wx + B * wy * wz;
    Rt[8] = -A * wy + B * wx * wz;      Rt[9] = A * wx + B * wy * wz;       Rt[10] = 1.0 + B * (wz * wz - th2);
    double a[3], b[3];
    d3cross(phi, rho, a);
    d3cross(phi, a, b);
    Rt[3] = rho[0] + B * a[0] + C * b[0];
    Rt[7] = rho[1] + B * a[1] + C * b[1];
    Rt[11] = rho[2] + B * a[2] + C * b[2];
}

// What the scoring needs beside n hypotheses' own rows, by the first 32 of the threads:
// zeros as the partner of an odd last one, and the pixel chunks of a frame with few.
__device__ __forceinline__ void finish_hypotheses(const DevParams& p, const DevState& s, int n, int id)
{
    if (id >= 32) return;
    if ((n & 1) && id < kScHypChunks) clear_hyp_operand(s.sc_hyp, n, id);
    const int groups = (n + kScGroupHyps - 1) / kScGroupHyps, all = (p.S + kScGroupHyps - 1) / kScGroupHyps;
    int chunks = 0;
    if (groups > 0 && groups < all)
        chunks = chunks_for_groups(groups, max(1, (*s.pix_count + kScTilePix - 1) / kScTilePix), s.chunks_max, s.score_ctas);
    if (id == 0) *s.few_chunks = chunks;
}

// Hypothesis collection: four lanes per (group, solution slot), one for each row of
// [R | t], write its solution h = offset + slot < S with its scoring form and tensor-core operand.
// A block covers the 8 groups of a P3P chunk and finds its offset itself, from the chunks'
// and the coarse counts that P3P leaves (at most 255 and 128 of them): a scan kernel
// before this one took 4 us and a launch per frame, and the sum of all earlier groups'
// counts, G^2 / 16 of them in all, 0.4 of 2.0 ms of a frame with 262144 groups solved.
// A lane per solution, with all of its FP64 work, took 10.7 us at S = 256 (14.6 at
// 8192), four lanes with 32 groups to a block, all on one SM, 12.2 (19.1); now 7.7 (14.7).
constexpr int kHypGroups = kP3PChunk;      // groups per block
constexpr int kHypThreads = kHypGroups * kMaxSols * 4;

__global__ void __launch_bounds__(kHypThreads) k_hyp_write(DevParams p, DevState s, int t)
{
    __shared__ int wsum[kHypThreads / 32], off_s[kHypGroups], n_s;
    __shared__ double e0[12];
    const int tid = threadIdx.x, lane = tid & 31;
    const bool current = *s.sc_ref != 0;
    const int G = groups_solved(p, s), g0 = blockIdx.x * kHypGroups;
    if (g0 >= G && blockIdx.x > 0) return;
    const double q = p.fyd / p.fxd;
    const double sc[3] = {1.0, q, 1.0};
    if (tid < 12) {                                       // the frame's reference pose in scaled form, {E, t}
        const double* T0 = s.poses + 12 * (t - 1);
        const int r = tid < 9 ? tid / 3 : tid - 9, c = tid < 9 ? tid % 3 : 3;
        double v = T0[r * 4 + c] - (r == c ? 1.0 : 0.0);
        if (q != 1.0) v = c < 3 ? sc[r] * v / sc[c] : sc[r] * v;     // square pixels need no scaling
        e0[r * 4 + c] = current ? v : 0.0;
    }
    int before = 0;
    const int full = blockIdx.x / kP3PBlock;              // coarse counts before this block's groups
    for (int i = tid; i < full; i += kHypThreads) before += s.block_sols[i];
    for (int i = full * kP3PBlock + tid; i < blockIdx.x; i += kHypThreads) before += s.chunk_sols[i];
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
    if (lane == 0) wsum[tid >> 5] = before;
    __syncthreads();
    if (tid < 32) {
        int base = 0;
        for (int w = 0; w < kHypThreads / 32; ++w) base += wsum[w];
        const int c = tid < kHypGroups && g0 + tid < G ? s.grp_count[g0 + tid] : 0;
        int incl = c;
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (tid < kHypGroups) off_s[tid] = base + incl - c;
        if (tid == 31) {
            n_s = -1;
            if (g0 + kHypGroups >= G) *s.n_hyp = n_s = min(base + incl, p.S);      // the last block with groups
        }
    }
    __syncthreads();
    const int item = tid >> 2, r = min(tid & 3, 2), g = g0 + item / kMaxSols, i = item % kMaxSols;
    const int h = off_s[item / kMaxSols] + i;
    if (n_s >= 0) finish_hypotheses(p, s, n_s, kHypThreads - 1 - tid);    // the last warp, whose slots are seldom all filled
    if (g >= G || i >= s.grp_count[g] || h >= p.S) return;                // whole quads leave together
    const double* Rt = s.grp_sols + ((size_t)g * kMaxSols + i) * 12 + r * 4;
    double v[4], e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        v[c] = Rt[c];
        e[c] = v[c] - (r == c ? 1.0 : 0.0);
    }
    if (q != 1.0) {                        // square pixels need no scaling, and FP64 divisions are long here
        for (int c = 0; c < 3; ++c) e[c] = sc[r] * e[c] / sc[c];
        e[3] = sc[r] * e[3];
    }
    if ((tid & 3) < 3) {
        double* oR = s.hyp_Rt + (size_t)h * 12;
        float* f = s.hyp_f32 + (size_t)h * 12;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            oR[c < 3 ? r * 3 + c : 9 + r] = v[c];
            f[c < 3 ? r * 3 + c : 9 + r] = (float)e[c];
        }
    } else {
        s.hyp_w[h] = s.grp_weight[g];
        s.hyp_info[(size_t)h * 2 + 0] = g;
        s.hyp_info[(size_t)h * 2 + 1] = i;
    }
    if (write_hyp_operand(s.sc_hyp, h, e, e0 + 4 * r)) atomicOr(s.sc_wild, 1);
}

// The meanshift's form of hypothesis h (after k_hyp_write): its se(3)
// logarithm, each coordinate as a float-float pair (hi = v rounded, lo =
// v - hi rounded), and its weight in FP32. A long FP64 chain per hypothesis,
// needed only by the meanshift: it runs on a side branch beside the scoring.
__global__ void k_hyp_log(DevParams p, DevState s)
{
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= *s.n_hyp) return;
    const long long g = s.hyp_info[(size_t)h * 2 + 0], i = s.hyp_info[(size_t)h * 2 + 1];
    double pv[6];
    se3_log_quat(s.grp_sols + ((size_t)g * kMaxSols + i) * 12, pv);
    float hi[6], lo[6];
    for (int c = 0; c < 6; ++c) {
        hi[c] = (float)pv[c];
        lo[c] = (float)(pv[c] - (double)hi[c]);
    }
    float4* pw = reinterpret_cast<float4*>(s.hyp_pw + (size_t)h * 16);
    pw[0] = make_float4(hi[0], hi[1], hi[2], hi[3]);
    pw[1] = make_float4(hi[4], hi[5], lo[0], lo[1]);
    pw[2] = make_float4(lo[2], lo[3], lo[4], lo[5]);
    pw[3] = make_float4((float)s.hyp_w[h], 0.f, 0.f, 0.f);
}

void launch_hyp_log(const DevParams& p, const DevState& s, cudaStream_t st)
{
    k_hyp_log<<<(p.S + 127) / 128, 128, 0, st>>>(p, s);
}

void launch_hyp_collect(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    // sized for the budget; blocks past the solved prefix return at once
    k_hyp_write<<<(p.G + kHypGroups - 1) / kHypGroups, kHypThreads, 0, st>>>(p, s, t);
}

// Scoring form of caller-given hypotheses already copied to hyp_Rt.
__global__ void k_hyp_from_rt(DevParams p, DevState s, int t, int n)
{
    const int id = blockIdx.x * blockDim.x + threadIdx.x, h = id >> 2, r = min(id & 3, 2);
    if (id == 0) *s.n_hyp = n;
    finish_hypotheses(p, s, n, id);
    if (h >= n) return;                                   // whole quads leave together
    const double q = p.fyd / p.fxd;
    const double sc[3] = {1.0, q, 1.0};
    const double* R = s.hyp_Rt + (size_t)h * 12;
    const double* T0 = s.poses + 12 * (t - 1) + r * 4;
    double e[4], e0[4];
    for (int c = 0; c < 3; ++c) {
        e[c] = sc[r] * (R[r * 3 + c] - (r == c ? 1.0 : 0.0)) / sc[c];
        e0[c] = *s.sc_ref ? sc[r] * (T0[c] - (r == c ? 1.0 : 0.0)) / sc[c] : 0.0;
    }
    e[3] = sc[r] * R[9 + r];
    e0[3] = *s.sc_ref ? sc[r] * T0[3] : 0.0;
    if ((id & 3) < 3) {
        float* f = s.hyp_f32 + (size_t)h * 12;
        for (int c = 0; c < 4; ++c) f[c < 3 ? r * 3 + c : 9 + r] = (float)e[c];
    }
    if (write_hyp_operand(s.sc_hyp, h, e, e0)) atomicOr(s.sc_wild, 1);
}

void score_hyps_from_host(const DevParams& p, const DevState& s, int t, int n, cudaStream_t st)
{
    k_hyp_from_rt<<<(4 * n + 127) / 128 + 1, 128, 0, st>>>(p, s, t, n);
}

// ---------------------------------------------------------------------------
// Meanshift (Eqs. 18-19): x <- sum_h w_h K(x - p_h) p_h / sum_h w_h K(x - p_h),
// K(d) = exp(-d^T Sigma^-1 d / 2), seeded at argmax_h L_h (lowest index on
// ties), on a cluster of kMeanshiftCtas CTAs. Everything runs on the FP32
// pipe (an FP64 instruction is a long issue on this GPU's FP64 pipe, and this
// kernel is a chain of small dependent steps): the argmax compares the FP64
// scores as order-preserving integer keys; each hypothesis is held as its
// FP32 offset from the seed, taken from float-float copies of the se(3)
// logarithms, so the Gaussian and the per-thread partial sums are FP32 on
// small numbers; sums across warps and CTAs and the state (the offset of x
// from the seed) are float-float, about 44 significant bits. Every CTA
// reduces the cluster's partial sums in the same order, so all take the same
// steps; partial buffers alternate by iteration parity so one cluster barrier
// per step suffices, and one warp finishes the step (sums across CTAs, new
// state, convergence) with shuffles. The iteration stops when the step is
// below ms_tol, when a step below 1e-7 no longer contracts (the FP32 noise
// floor of the kernel weights), or after ms_max_iter steps.
// ---------------------------------------------------------------------------
constexpr int kMsCached = 4;     // hypotheses per thread held in registers (all of them up to S = 8192)

// Order-preserving integer key of a double: a < b iff key(a) < key(b) for
// non-NaN values, -0 and +0 equal.
__device__ __forceinline__ long long score_key(double v)
{
    long long b = __double_as_longlong(v);
    if (b == (long long)0x8000000000000000ull) b = 0;
    return b >= 0 ? b : (b ^ 0x7fffffffffffffffll);
}

// The frame tables after the pose update of frame t: C_t = T_t C_{t-1} and T_t in the
// forms k_frame_setup writes, with the same operations (products and sums rounded
// one by one, so the values are bit-identical to a set-up from scratch). One CTA,
// after poses[t - 1] is written: a set-up kernel before every frame and stage cost
// 5-8 us each, most of it the FP64 chain over all frames.
__device__ void advance_frame_tables(const DevParams& p, const DevState& s, int t)
{
    __shared__ double T[12], C[12];
    const int i = threadIdx.x;
    __syncthreads();
    if (i < 12) {
        T[i] = s.poses[12 * (t - 1) + i];
        C[i] = s.cum[12 * (t - 1) + i];
    }
    __syncthreads();
    if (i >= 12) return;
    const int r = i / 4, c = i % 4;
    const double one = r == c ? 1.0 : 0.0;
    const double av = T[i];
    double cv = __dadd_rn(__dadd_rn(__dmul_rn(T[4 * r], C[c]), __dmul_rn(T[4 * r + 1], C[4 + c])),
                          __dmul_rn(T[4 * r + 2], C[8 + c]));
    if (c == 3) cv = __dadd_rn(cv, T[4 * r + 3]);
    const float ah = (float)av, ch = (float)cv;
    s.poses_df[24 * (t - 1) + 2 * i] = ah;
    s.poses_df[24 * (t - 1) + 2 * i + 1] = (float)(av - (double)ah);
    s.frames32[24 * (t - 1) + 12 + (c < 3 ? 3 * r + c : 9 + r)] = c < 3 ? (float)(av - one) : ah;
    if (t == p.T) return;
    s.cum[12 * t + i] = cv;
    s.cum_df[24 * t + 2 * i] = ch;
    s.cum_df[24 * t + 2 * i + 1] = (float)(cv - (double)ch);
    s.frames32[24 * t + (c < 3 ? 3 * r + c : 9 + r)] = c < 3 ? (float)(cv - one) : ch;
}

__device__ __forceinline__ DF shfl_df(DF v, int src)
{
    return DF{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}

// Sums of eight per-lane values over a warp: at each step a lane keeps half of its
// values and adds the partner's, so lane l ends with the sum of value l / 4 (9 shuffles
// instead of 5 per value). The pairs are those of an xor butterfly from 16 down to
// 1, so each sum is bit-identical to it.
__device__ __forceinline__ float warp_sum8(const float* a, int lane)
{
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const bool up = (lane & 16) != 0;
        v[i] = (up ? a[i + 4] : a[i]) + __shfl_xor_sync(0xffffffffu, up ? a[i] : a[i + 4], 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const bool up = (lane & 8) != 0;
        v[i] = (up ? v[i + 2] : v[i]) + __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + 2], 8);
    }
    const bool up = (lane & 4) != 0;
    float r = (up ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, up ? v[0] : v[1], 4);
    r += __shfl_xor_sync(0xffffffffu, r, 2);
    return r + __shfl_xor_sync(0xffffffffu, r, 1);
}

// Shared state of a meanshift CTA.
struct MsShared {
    float wred[32][8];                    // the warps' sums of the step
    float2 part[2][8];                    // the CTA's sums, by step parity (cluster form)
    float xo_hi[6], xo_lo[6];             // x - p_seed, float-float
    float seed_hi[6], seed_lo[6];
    long long bkey[32];
    int bidx[32];
    int flag;
    float consts[3];
};

// argmax of L (lowest index on ties; NaN never wins), then the seed and the
// constants into shared memory. Eight scores in flight per thread.
__device__ __forceinline__ void ms_seed(const DevParams& p, const DevState& s, MsShared& m, int n)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    long long bk = 0;
    int bi = 0x7fffffff;
    for (int h0 = tid; h0 < n; h0 += 8 * blockDim.x) {
        double v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = h0 + i * (int)blockDim.x < n ? s.scores[h0 + i * blockDim.x] : NAN;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const long long raw = __double_as_longlong(v[i]) & 0x7fffffffffffffffll;
            if (raw > 0x7ff0000000000000ll) continue;             // NaN
            const long long k = score_key(v[i]);
            if (bi == 0x7fffffff || k > bk) { bk = k; bi = h0 + i * blockDim.x; }   // increasing h: the first wins ties
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (oi != 0x7fffffff && (bi == 0x7fffffff || ok > bk || (ok == bk && oi < bi))) { bk = ok; bi = oi; }
    }
    if (lane == 0) { m.bkey[warp] = bk; m.bidx[warp] = bi; }
    __syncthreads();
    if (warp == 0) {
        bk = lane < nwarp ? m.bkey[lane] : 0;
        bi = lane < nwarp ? m.bidx[lane] : 0x7fffffff;
        for (int o = 16; o > 0; o >>= 1) {
            const long long ok = __shfl_xor_sync(0xffffffffu, bk, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (oi != 0x7fffffff && (bi == 0x7fffffff || ok > bk || (ok == bk && oi < bi))) { bk = ok; bi = oi; }
        }
        if (bi == 0x7fffffff) bi = 0;
        if (lane < 6) {
            const float* ps = s.hyp_pw + (size_t)bi * 16;
            m.seed_hi[lane] = ps[lane];
            m.seed_lo[lane] = ps[6 + lane];
            m.xo_hi[lane] = 0.f;
            m.xo_lo[lane] = 0.f;
        }
        if (lane == 6) m.bidx[0] = bi;
        if (lane == 7) m.flag = 0;
    } else if (tid == 32) {
        m.consts[0] = (float)(1.0 / p.sigma_t);
        m.consts[1] = (float)(1.0 / p.sigma_r);
        m.consts[2] = (float)p.ms_tol;
    }
    __syncthreads();
}

// Offset of hypothesis h from the seed in FP32, its weight in o1.z.
__device__ __forceinline__ void ms_offset(const DevState& s, const DF* sd, int h, float4& o0, float4& o1)
{
    const float4* pw = reinterpret_cast<const float4*>(s.hyp_pw + (size_t)h * 16);
    const float4 a = pw[0], b = pw[1], c2 = pw[2], d = pw[3];
    const float ph[6] = {a.x, a.y, a.z, a.w, b.x, b.y}, pl[6] = {b.z, b.w, c2.x, c2.y, c2.z, c2.w};
    float o[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) o[c] = df_to_float(df_sub(DF{ph[c], pl[c]}, sd[c]));
    o0 = make_float4(o[0], o[1], o[2], o[3]);
    o1 = make_float4(o[4], o[5], d.x, 0.f);
}

// acc += w K(x - p) (1, p) for one offset.
__device__ __forceinline__ void ms_add(const float* dx, float ivt, float ivr, const float4 q0, const float4 q1, float* acc)
{
    const float mlog2e = -0.5f * 1.4426950408889634f;
    const float d0 = dx[0] - q0.x, d1 = dx[1] - q0.y, d2 = dx[2] - q0.z;
    const float d3 = dx[3] - q0.w, d4 = dx[4] - q1.x, d5 = dx[5] - q1.y;
    const float m = fmaf(d0 * d0 + d1 * d1 + d2 * d2, ivt, (d3 * d3 + d4 * d4 + d5 * d5) * ivr);
    const float kw = q1.z * exp2f(mlog2e * m);
    if (!(kw > 0.f)) return;       // zero weight (or a non-finite hypothesis) adds nothing
    acc[0] += kw;
    acc[1] = fmaf(kw, q0.x, acc[1]); acc[2] = fmaf(kw, q0.y, acc[2]); acc[3] = fmaf(kw, q0.z, acc[3]);
    acc[4] = fmaf(kw, q0.w, acc[4]); acc[5] = fmaf(kw, q1.x, acc[5]); acc[6] = fmaf(kw, q1.y, acc[6]);
}

// One warp finishes a step from the total (component c in lane c < 7): the new
// state, and the flag 0 go on, 1 converged, 2 no mass at the first step.
__device__ __forceinline__ void ms_finish(MsShared& m, DF tot, int lane, int it, float tol, float& prev_step)
{
    const DF t0 = shfl_df(tot, 0);
    const bool mass = t0.hi > 0.f;
    float dd = 0.f;
    if (mass && lane >= 1 && lane < 7) {
        const DF xn = df_div(tot, t0);                    // mean offset of component lane - 1
        const DF xo{m.xo_hi[lane - 1], m.xo_lo[lane - 1]};
        dd = df_to_float(df_sub(xn, xo));
        dd *= dd;
        m.xo_hi[lane - 1] = xn.hi;
        m.xo_lo[lane - 1] = xn.lo;
    }
    float s2 = 0.f;
#pragma unroll
    for (int c = 1; c < 7; ++c) s2 += __shfl_sync(0xffffffffu, dd, c);
    if (lane == 0) {
        if (!mass) {
            m.flag = (it == 0) ? 2 : 1;
        } else {
            const float step = sqrtf(s2);
            m.flag = (step < tol || (step >= prev_step && step < 1e-7f)) ? 1 : 0;
            prev_step = step;
        }
    }
}

// Status words, the pose and the frame tables (one CTA).
__device__ __forceinline__ void ms_result(const DevParams& p, const DevState& s, const MsShared& m, int t, int n, int seed,
                                          int it, bool degenerate)
{
    if (threadIdx.x == 0) {
        s.status[0] = n;
        s.status[1] = seed;
        s.status[2] = it;
        if (degenerate) {
            s.status[3] += 1;
        } else {
            double x[6];
            for (int c = 0; c < 6; ++c)
                x[c] = ((double)m.seed_hi[c] + (double)m.seed_lo[c]) + ((double)m.xo_hi[c] + (double)m.xo_lo[c]);
            se3_exp_vec(x, s.poses + 12 * (t - 1));
        }
    }
    advance_frame_tables(p, s, t);
}

__device__ __forceinline__ void ms_no_hypothesis(const DevParams& p, const DevState& s, int t)
{
    if (threadIdx.x == 0) {
        s.status[0] = 0; s.status[1] = -1; s.status[2] = 0; s.status[3] += 1;
    }
    advance_frame_tables(p, s, t);        // the pose stays, but C_{t-1} may have moved
}

// A cluster of kMeanshiftCtas CTAs, hypothesis h in CTA (h / 256) % 8.
__global__ void __cluster_dims__(kMeanshiftCtas, 1, 1) __launch_bounds__(kMeanshiftThreads, 1)
k_meanshift(DevParams p, DevState s, int t)
{
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned rank = cluster.block_rank();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    __shared__ MsShared m;
    const int n = *s.n_hyp;
    if (n == 0) {
        if (rank == 0) ms_no_hypothesis(p, s, t);
        return;   // uniform over the cluster: every CTA reads the same n
    }
    ms_seed(p, s, m, n);
    const int seed = m.bidx[0];
    // FP32 offsets of this CTA's hypotheses from the seed: a thread's first
    // kMsCached stay in registers, the rest (S above kMsCached x the cluster's
    // threads) go to global memory
    const int stride = kMeanshiftCtas * blockDim.x, h0 = rank * blockDim.x + tid;
    DF sd[6];
    for (int c = 0; c < 6; ++c) sd[c] = DF{m.seed_hi[c], m.seed_lo[c]};
    float4 r0[kMsCached], r1[kMsCached];
#pragma unroll
    for (int k = 0; k < kMsCached; ++k) {
        r0[k] = r1[k] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (h0 + k * stride < n) ms_offset(s, sd, h0 + k * stride, r0[k], r1[k]);
    }
    for (int h = h0 + kMsCached * stride; h < n; h += stride) {
        float4* od = reinterpret_cast<float4*>(s.hyp_dp + (size_t)h * 8);
        ms_offset(s, sd, h, od[0], od[1]);
    }
    const float ivt = m.consts[0], ivr = m.consts[1], tol = m.consts[2];
    int it = 0;
    bool degenerate = false;
    float prev_step = INFINITY;
    for (; it < p.ms_max_iter; ++it) {
        float dx[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) dx[c] = m.xo_hi[c] + m.xo_lo[c];
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        // hypotheses in increasing h (the registers' first, then global memory)
#pragma unroll
        for (int k = 0; k < kMsCached; ++k)
            if (h0 + k * stride < n) ms_add(dx, ivt, ivr, r0[k], r1[k], acc);
        for (int h = h0 + kMsCached * stride; h < n; h += stride) {
            const float4* o = reinterpret_cast<const float4*>(s.hyp_dp + (size_t)h * 8);
            ms_add(dx, ivt, ivr, o[0], o[1], acc);
        }
        // warp sums in FP32 (each lane holds at most 4 terms), then the CTA's
        // warps in order as float-float
        const float ws = warp_sum8(acc, lane);
        if ((lane & 3) == 0) m.wred[warp][lane >> 2] = ws;
        __syncthreads();
        const int buf = it & 1;
        if (tid < 7) {
            DF v{0.f, 0.f};
            for (int w = 0; w < nwarp; ++w) v = df_add(v, m.wred[w][tid]);
            m.part[buf][tid] = make_float2(v.hi, v.lo);
        }
        cluster.sync();
        if (warp == 0) {
            // lane c < 7 adds component c of the ranks' sums in rank order, all
            // eight loads from distributed shared memory in flight at once
            float2 g[kMeanshiftCtas];
#pragma unroll
            for (int r = 0; r < kMeanshiftCtas; ++r)
                g[r] = lane < 7 ? *cluster.map_shared_rank(&m.part[buf][lane], (unsigned)r) : make_float2(0.f, 0.f);
            DF tot{0.f, 0.f};
#pragma unroll
            for (int r = 0; r < kMeanshiftCtas; ++r) tot = df_add(tot, DF{g[r].x, g[r].y});
            ms_finish(m, tot, lane, it, tol, prev_step);
        }
        __syncthreads();
        const int f = m.flag;
        if (f == 2) { degenerate = true; break; }
        if (f == 1) { ++it; break; }
    }
    cluster.sync();   // no CTA leaves while another may still read its partials
    if (rank == 0) ms_result(p, s, m, t, n, seed, it, degenerate);
}

// The same for at most 1024 hypotheses in one CTA, one hypothesis per thread: no
// cluster barrier and no distributed shared memory in the step. The sums keep the
// cluster form's order (eight warps of 256 hypotheses, then those groups), so the
// result is bit-identical to it.
constexpr int kMsBlockMax = 1024;

__global__ void __launch_bounds__(kMsBlockMax, 1) k_meanshift_block(DevParams p, DevState s, int t)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, groups = blockDim.x / kMeanshiftThreads;
    __shared__ MsShared m;
    const int n = *s.n_hyp;
    if (n == 0) {
        ms_no_hypothesis(p, s, t);
        return;
    }
    ms_seed(p, s, m, n);
    const int seed = m.bidx[0];
    DF sd[6];
    for (int c = 0; c < 6; ++c) sd[c] = DF{m.seed_hi[c], m.seed_lo[c]};
    float4 r0 = make_float4(0.f, 0.f, 0.f, 0.f), r1 = r0;
    if (tid < n) ms_offset(s, sd, tid, r0, r1);
    const float ivt = m.consts[0], ivr = m.consts[1], tol = m.consts[2];
    int it = 0;
    bool degenerate = false;
    float prev_step = INFINITY;
    for (; it < p.ms_max_iter; ++it) {
        float dx[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) dx[c] = m.xo_hi[c] + m.xo_lo[c];
        float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        if (tid < n) ms_add(dx, ivt, ivr, r0, r1, acc);
        const float ws = warp_sum8(acc, lane);
        if ((lane & 3) == 0) m.wred[warp][lane >> 2] = ws;
        __syncthreads();
        if (warp == 0) {
            // lane 8 g + c: component c of group g's eight warps in order, then the groups in order
            const int g = lane >> 3, c = lane & 7;
            DF v{0.f, 0.f};
            if (g < groups)
                for (int w = 0; w < 8; ++w) v = df_add(v, m.wred[8 * g + w][c]);
            DF tot{0.f, 0.f};
            for (int r = 0; r < groups; ++r) tot = df_add(tot, shfl_df(v, 8 * r + c));
            ms_finish(m, tot, lane, it, tol, prev_step);
        }
        __syncthreads();
        const int f = m.flag;
        if (f == 2) { degenerate = true; break; }
        if (f == 1) { ++it; break; }
    }
    ms_result(p, s, m, t, n, seed, it, degenerate);
}

// Up to 1024 hypotheses fit one CTA.
void launch_meanshift(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    if (p.S <= kMsBlockMax) {
        const int threads = (p.S + kMeanshiftThreads - 1) / kMeanshiftThreads * kMeanshiftThreads;
        k_meanshift_block<<<1, threads, 0, st>>>(p, s, t);
    } else {
        k_meanshift<<<kMeanshiftCtas, kMeanshiftThreads, 0, st>>>(p, s, t);
    }
}

}  // namespace vd
