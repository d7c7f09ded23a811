// Per-pixel kernels of the VOLDOR loop: frame pose setup, bootstrap
// triangulation and the MIE depth sweep (the FP64-geometry passes are in
// k_geom.cu).
//
// This translation unit is compiled without FMA contraction (--fmad=false):
// the MIE sweep compares a candidate scored in one kernel with one scored in
// another, and equal depths must give bit-identical scores.
#include "df32.cuh"
#include "voldor_internal.cuh"

namespace vd {

// ---------------------------------------------------------------------------
// Frame setup: C_{t-1} = T_{t-1} ... T_1 for every t (FP64), the product of
// Eq. 1 with T_t the motion from t-1 to t.
// ---------------------------------------------------------------------------
// The poses are staged in shared memory, then lane 4 r + c of the first warp carries
// element (r, c) of C (O = A C: O[r, c] = A[r, :3] C[:, c], plus A's translation for
// c = 3), each element added in the same order as the row-by-row product. A lane per
// column took three times the FP64 instructions: 8.5 us at T = 8, now 5.2.
__global__ void k_frame_setup(DevParams p, DevState s)
{
    __shared__ double A[kMaxT * 12];
    __shared__ double Cs[kMaxT * 12];          // C_{t-1}, [t - 1][3][4]
    for (int i = threadIdx.x; i < p.T * 12; i += blockDim.x) A[i] = s.poses[i];
    __syncthreads();
    // the product chain C_t = T_t C_{t-1}
    if (threadIdx.x < 12) {
        const int i = threadIdx.x, r = i / 4, c = i % 4;
        double C = r == c ? 1.0 : 0.0;
        for (int t = 1; t <= p.T; ++t) {
            Cs[12 * (t - 1) + i] = C;
            const double* At = A + 12 * (t - 1) + 4 * r;
            const double C0 = __shfl_sync(0xfffu, C, c), C1 = __shfl_sync(0xfffu, C, 4 + c), C2 = __shfl_sync(0xfffu, C, 8 + c);
            C = At[0] * C0 + At[1] * C1 + At[2] * C2;
            if (c == 3) C = C + At[3];
        }
    }
    __syncthreads();
    // every stage's outputs, one element (t, r, col) per thread: C_{t-1} in FP64
    // and as float-float pairs (hi = fl32(v), lo = fl32(v - hi)), T_t as
    // float-float pairs, and both as E = R - I, t in FP32
    for (int i = threadIdx.x; i < p.T * 12; i += blockDim.x) {
        const int t1 = i / 12, e = i % 12, r = e / 4, col = e % 4;
        const double cv = Cs[i], av = A[i];
        s.cum[i] = cv;
        const float ch = (float)cv, ah = (float)av;
        s.cum_df[2 * i] = ch;
        s.cum_df[2 * i + 1] = (float)(cv - (double)ch);
        s.poses_df[2 * i] = ah;
        s.poses_df[2 * i + 1] = (float)(av - (double)ah);
        float* f = s.frames32 + 24 * t1;        // E_c = R_c - I, t_c, E_t = R_t - I, t_t
        if (col < 3) {
            f[3 * r + col] = (float)(cv - (r == col ? 1.0 : 0.0));
            f[12 + 3 * r + col] = (float)(av - (r == col ? 1.0 : 0.0));
        } else {
            f[9 + r] = (float)cv;
            f[21 + r] = (float)av;
        }
    }
}

void launch_frame_setup(const DevParams& p, const DevState& s, cudaStream_t st)
{
    k_frame_setup<<<1, kMaxT * 12, 0, st>>>(p, s);
}

// ---------------------------------------------------------------------------
// Bootstrap (Table 1): W := 1, poses := T_1, k := 0, and per pixel the
// least-squares depth along the ray of pixel j from x_j + X_1^j ~ pi_1(theta).
// With d = K^-1 [x y 1], m = K^-1 [x+u y+v 1]:
//   a_x = (R d)_x - m_x (R d)_z,  b_x = m_x t_z - t_x  (same for y),
//   theta = (a.b)/(a.a), i.e. inverse depth (a.a)/(a.b), clamped; the result
//   is that of FP64.
// ---------------------------------------------------------------------------
struct BootPose {
    double T[12];
    DF Td[12];              // the same as float-float pairs
    float far32, near32;    // the FP32 depths of the clamps, 1 / inv_depth_min and 1 / inv_depth_max
};

// The depth in FP64 (the definition).
__device__ __noinline__ float bootstrap_depth64(const DevParams& p, const double* M, int x, int y, float2 f)
{
    const double dx = ((double)x - p.cxd) * p.inv_fxd, dy = ((double)y - p.cyd) * p.inv_fyd;
    const double mx = ((double)x + f.x - p.cxd) * p.inv_fxd, my = ((double)y + f.y - p.cyd) * p.inv_fyd;
    const double Rdx = M[0] * dx + M[1] * dy + M[2];
    const double Rdy = M[4] * dx + M[5] * dy + M[6];
    const double Rdz = M[8] * dx + M[9] * dy + M[10];
    const double ax = Rdx - mx * Rdz, bx = mx * M[11] - M[3];
    const double ay = Rdy - my * Rdz, by = my * M[11] - M[7];
    const double num = ax * ax + ay * ay, den = ax * bx + ay * by;
    double inv = (double)p.inv_depth_min;
    if (den > 0.0) {
        const double r = num / den;
        if (isfinite(r)) inv = fmin(fmax(r, (double)p.inv_depth_min), (double)p.inv_depth_max);
    }
    return (float)(1.0 / inv);
}

// The same FP32 depth through float-float arithmetic beside a bound of its error;
// false where the bound leaves the sign of a.b, the clamp or the last bit open.
// In units of 2^-48: a sum errs by 2 of its terms' magnitudes, a product by 6, a
// pair made of an FP64 constant by 1/2; so m and d by 9, R d by 20, a by 37 and b by
// 18 of the sums of their terms' magnitudes, taken as 40 and 20.
__device__ __forceinline__ bool bootstrap_depth32(const DevParams& p, const BootPose& bp, int x, int y, float2 f, float& depth)
{
    const DF* M = bp.Td;
    const DF cx{p.kdf[4], p.kdf[5]}, cy{p.kdf[6], p.kdf[7]}, ifx{p.kdf[8], p.kdf[9]}, ify{p.kdf[10], p.kdf[11]};
    const float xf = (float)x, yf = (float)y;
    const DF dx = df_mul(df_add(df_neg(cx), xf), ifx), dy = df_mul(df_add(df_neg(cy), yf), ify);
    const DF mx = df_mul(df_sub(df_two_sum(xf, f.x), cx), ifx), my = df_mul(df_sub(df_two_sum(yf, f.y), cy), ify);
    const DF Rx = df_add(df_add(df_mul(M[0], dx), df_mul(M[1], dy)), M[2]);
    const DF Ry = df_add(df_add(df_mul(M[4], dx), df_mul(M[5], dy)), M[6]);
    const DF Rz = df_add(df_add(df_mul(M[8], dx), df_mul(M[9], dy)), M[10]);
    const DF ax = df_sub(Rx, df_mul(mx, Rz)), bx = df_sub(df_mul(mx, M[11]), M[3]);
    const DF ay = df_sub(Ry, df_mul(my, Rz)), by = df_sub(df_mul(my, M[11]), M[7]);
    const DF num = df_add(df_mul(ax, ax), df_mul(ay, ay)), den = df_add(df_mul(ax, bx), df_mul(ay, by));

    const float ux = (xf + fabsf(cx.hi)) * ifx.hi, uy = (yf + fabsf(cy.hi)) * ify.hi;
    const float vx = ux + fabsf(f.x) * ifx.hi, vy = uy + fabsf(f.y) * ify.hi;
    const float sx = fabsf(M[0].hi) * ux + fabsf(M[1].hi) * uy + fabsf(M[2].hi);
    const float sy = fabsf(M[4].hi) * ux + fabsf(M[5].hi) * uy + fabsf(M[6].hi);
    const float sz = fabsf(M[8].hi) * ux + fabsf(M[9].hi) * uy + fabsf(M[10].hi);
    const float eax = 40.f * 0x1p-48f * (sx + vx * sz), ebx = 20.f * 0x1p-48f * (vx * fabsf(M[11].hi) + fabsf(M[3].hi));
    const float eay = 40.f * 0x1p-48f * (sy + vy * sz), eby = 20.f * 0x1p-48f * (vy * fabsf(M[11].hi) + fabsf(M[7].hi));
    const float aax = fabsf(ax.hi) + eax, aay = fabsf(ay.hi) + eay, abx = fabsf(bx.hi) + ebx, aby = fabsf(by.hi) + eby;
    const float e_den = aax * ebx + abx * eax + aay * eby + aby * eay + 8.f * 0x1p-48f * (aax * abx + aay * aby);
    const float e_num = 2.f * (aax * eax + aay * eay) + 8.f * 0x1p-48f * num.hi;
    if (den.hi < -e_den) {
        depth = bp.far32;
        return true;
    }
    if (!(den.hi > 1e-25f && num.hi > 1e-25f)) return false;
    const float rel = 1.01f * (__fdividef(e_den, den.hi) + __fdividef(e_num, num.hi)) + 32.f * 0x1p-48f;      // the last: the quotient's
    if (!(rel < 0x1p-24f)) return false;
    const float q = __fdividef(den.hi, num.hi);
    const float l = __fdividef(df_sub(den, df_mul(num, q)).hi, num.hi), err = q * rel;
    const float lo = __fadd_rn(q, l - err), hi = __fadd_rn(q, l + err);
    constexpr float kOut = 1.f + 0x1p-20f, kIn = 1.f - 0x1p-20f;
    if (hi < bp.near32 * kIn) depth = bp.near32;
    else if (lo > bp.far32 * kOut) depth = bp.far32;
    else if (lo == hi && lo > bp.near32 * kOut && lo < bp.far32 * kIn) depth = lo;
    else return false;
    return true;
}

// In FP64 alone (66 FP64 instructions a pixel, two of them divisions) this took
// 56 us at 1242 x 375; now 15.7 us.
__global__ void k_bootstrap(DevParams p, DevState s, BootPose bp)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j == 0) {
        for (int t = 0; t < p.T; ++t)
            for (int q = 0; q < 12; ++q) s.poses[12 * t + q] = bp.T[q];
        *s.iter = 0;
    }
    if (j >= p.N) return;
    for (int t = 0; t < p.T; ++t) s.wmap[(size_t)t * p.N + j] = 1.f;
    const int x = j % p.W, y = j / p.W;
    const float2 f = load_flow(s.flows, p.flow_f16, (size_t)j);
    float depth;
    if (!bootstrap_depth32(p, bp, x, y, f, depth)) depth = bootstrap_depth64(p, bp.T, x, y, f);
    s.theta[j] = depth;
}

void launch_bootstrap(const DevParams& p, const DevState& s, const double* T1, cudaStream_t st)
{
    BootPose bp;
    for (int q = 0; q < 12; ++q) {
        bp.T[q] = T1[q];
        bp.Td[q].hi = (float)T1[q];
        bp.Td[q].lo = (float)(T1[q] - (double)bp.Td[q].hi);
    }
    bp.far32 = (float)(1.0 / (double)p.inv_depth_min);
    bp.near32 = (float)(1.0 / (double)p.inv_depth_max);
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    k_bootstrap<<<nb, kPixThreads, 0, st>>>(p, s, bp);
}


// ell_t(j) at depth d in FP32 for the MIE candidate scores, written without
// cancellation: with d = K^-1 [x y 1], the point in camera t-1 is
// theta (d + a), a = E_c d + t_c / theta, so pi_{t-1} = (x, y) + delta with
// delta = f (a_xy - d_xy a_z) / (1 + a_z) (a small quantity); the sample
// position is split into an integer pixel and a fraction; the rigid flow is
// xi = f (b_xy - pb_xy b_z) / (1 + b_z) with b = E_t pb + t_t / P_z. Every
// MIE candidate is scored by this one function, so equal depths score
// bit-identically.
struct FramesF {
    float v[kMaxT][24];
};

__device__ __forceinline__ void load_frames32(const DevParams& p, const DevState& s, FramesF& f)
{
    for (int i = threadIdx.x; i < p.T * 24; i += blockDim.x) f.v[i / 24][i % 24] = s.frames32[i];
    __syncthreads();
}

__device__ __forceinline__ float depth_ell_fast(const DevParams& p, const float* fr, const void* flows, int t, int x,
                                                int y, float depth)
{
    // invalid (t, j): rho := mu, i.e. log 1/2 under MIE and 0 under MLE
    const float ln_half = p.criterion == VOLDOR_CRITERION_MLE ? 0.f : -0.69314718055994531f;
    if (!(depth > 0.f)) return ln_half;
    const float dx = ((float)x - p.cx) * p.inv_fx, dy = ((float)y - p.cy) * p.inv_fy;
    const float w0 = 1.f / depth;
    float pbx = dx, pby = dy, w = w0;
    int x0 = x, y0 = y;
    float fxr = 0.f, fyr = 0.f;
    if (t > 1) {
        const float* E = fr;
        const float ax = fmaf(E[0], dx, fmaf(E[1], dy, fmaf(fr[9], w0, E[2])));
        const float ay = fmaf(E[3], dx, fmaf(E[4], dy, fmaf(fr[10], w0, E[5])));
        const float az = fmaf(E[6], dx, fmaf(E[7], dy, fmaf(fr[11], w0, E[8])));
        const float den = 1.f + az;
        if (!(den > 0.f)) return ln_half;
        const float rd = 1.f / den;
        const float mx = fmaf(-dx, az, ax) * rd, my = fmaf(-dy, az, ay) * rd;    // pb - d
        pbx = dx + mx;
        pby = dy + my;
        w = w0 * rd;
        const float du = p.fx * mx, dv = p.fy * my;     // pi_{t-1} - (x, y)
        if (!(fabsf(du) < 1e7f && fabsf(dv) < 1e7f)) return ln_half;
        const float iu = floorf(du), iv = floorf(dv);
        x0 = x + (int)iu;
        y0 = y + (int)iv;
        fxr = du - iu;
        fyr = dv - iv;
    }
    // valid iff 0 <= u <= W-1 and 0 <= v <= H-1
    if (x0 < 0 || y0 < 0 || x0 > p.W - 1 || y0 > p.H - 1) return ln_half;
    if ((x0 == p.W - 1 && fxr > 0.f) || (y0 == p.H - 1 && fyr > 0.f)) return ln_half;
    if (x0 == p.W - 1) { x0 = p.W - 2; fxr = 1.f; }
    if (y0 == p.H - 1) { y0 = p.H - 2; fyr = 1.f; }
    const size_t base = (size_t)(t - 1) * p.N + (size_t)y0 * p.W + x0;
    const float2 f00 = load_flow(flows, p.flow_f16, base), f10 = load_flow(flows, p.flow_f16, base + 1);
    const float2 f01 = load_flow(flows, p.flow_f16, base + p.W), f11 = load_flow(flows, p.flow_f16, base + p.W + 1);
    const float w00 = (1.f - fxr) * (1.f - fyr), w10 = fxr * (1.f - fyr), w01 = (1.f - fxr) * fyr, w11 = fxr * fyr;
    const float fu = fmaf(w00, f00.x, fmaf(w10, f10.x, fmaf(w01, f01.x, w11 * f11.x)));
    const float fv = fmaf(w00, f00.y, fmaf(w10, f10.y, fmaf(w01, f01.y, w11 * f11.y)));
    const float* Et = fr + 12;
    const float bx = fmaf(Et[0], pbx, fmaf(Et[1], pby, fmaf(fr[21], w, Et[2])));
    const float by = fmaf(Et[3], pbx, fmaf(Et[4], pby, fmaf(fr[22], w, Et[5])));
    const float bz = fmaf(Et[6], pbx, fmaf(Et[7], pby, fmaf(fr[23], w, Et[8])));
    const float den = 1.f + bz;
    if (!(den > 0.f)) return ln_half;
    const float rd = 1.f / den;
    const float ru = fmaf(p.fx * fmaf(-pbx, bz, bx), rd, -fu);
    const float rv = fmaf(p.fy * fmaf(-pby, bz, by), rd, -fv);
    const float xsq = fminf(fmaxf(fmaf(ru, ru, rv * rv), p.x_min), p.x_max);
    // MIE (Eq. 10): log rho/(rho+mu); MLE (Eq. 9): log rho - log mu
    return -neg_ell(p, xsq, sqrtf(fmaf(fu, fu, fv * fv)), p.criterion == VOLDOR_CRITERION_MLE);
}


// ---------------------------------------------------------------------------
// MIE depth update (Eq. 10, Fig. 5), chain-parallel with the exact sequential
// semantics. Along a chain, the sequential sweep carries one value v (the
// winner at the previous pixel) and at position i picks
//   v           if S_i(v) > S_i(prev_i) and S_i(v) >= S_i(smp_i),
//   own_i       otherwise, own_i = smp_i if S_i(smp_i) > S_i(prev_i) else prev_i,
// where S_i(d) = sum_t q_s(t, i) ell_t(i; d) summed in order t = 1..T. So the
// carried value is always own_r of the last position r where it was reset,
// and it survives from r until the first position where it loses. Three
// phases reproduce that bit for bit:
//   prepare  per pixel: S(prev), smp, S(smp), own;
//   runs     per pixel r (in parallel): test own_r at r+1, r+2, ... until it
//            loses, at most kRunCap positions (speculation);
//   resolve  per chain: follow r -> end of run from the chain start; a run
//            that reached the cap is continued there.
// ---------------------------------------------------------------------------
// Speculation pays where neighbouring pixels' tests share a warp's time, and costs where
// one lane of it goes on alone: runs + resolve take 43 + 110 us with a cap of 1, 71 + 89
// with 2, 98 + 79 with 3, 118 + 74 with 4 and 178 + 65 with 8 (the first four sweeps over a
// driving window of 1242 x 375, T = 8), and 30, 30, 29, 32 and 39 us together on 160 x 120.
constexpr int kRunCap = 2;

__device__ __forceinline__ float nan_to_ninf(float v) { return isnan(v) ? -INFINITY : v; }

__device__ __forceinline__ float mie_score(const DevParams& p, const DevState& s, const FramesF& f, int x, int y, float d)
{
    const int j = y * p.W + x;
    float acc = 0.f;
    for (int t = 1; t <= p.T; ++t) {
        const float q = s.qs[(size_t)(t - 1) * p.N + j];
        acc = __fadd_rn(acc, __fmul_rn(q, depth_ell_fast(p, f.v[t - 1], s.flows, t, x, y, d)));
    }
    return nan_to_ninf(acc);
}

// Under MIE no term of S is positive (log rho / (rho + mu), weights >= 0), so a partial
// sum only falls: once it is at most `limit` the whole is too. True if pixel j's
// weights allow that conclusion.
__device__ __forceinline__ bool falling(const DevParams& p, const DevState& s, int j)
{
    bool ok = p.criterion != VOLDOR_CRITERION_MLE;
    for (int t = 0; t < p.T; ++t) ok &= s.qs[(size_t)t * p.N + j] >= 0.f;
    return ok;
}

// S(d), or some partial sum at most `limit` where S(d) is at most `limit` too (then
// only that it loses against `limit` is of interest).
__device__ __forceinline__ float mie_score_above(const DevParams& p, const DevState& s, const FramesF& f, int x, int y, float d,
                                                 float limit)
{
    const int j = y * p.W + x;
    const bool stop = falling(p, s, j);
    float acc = 0.f;
    for (int t = 1; t <= p.T; ++t) {
        const float q = s.qs[(size_t)(t - 1) * p.N + j];
        acc = __fadd_rn(acc, __fmul_rn(q, depth_ell_fast(p, f.v[t - 1], s.flows, t, x, y, d)));
        if (stop && acc <= limit) break;
    }
    return nan_to_ninf(acc);
}

// Chain geometry: (x, y) of position i of chain c in direction dir.
__device__ __forceinline__ void chain_xy(const DevParams& p, int dir, int c, int i, int& x, int& y)
{
    switch (dir) {
        case 0: x = i; y = c; break;
        case 1: x = c; y = i; break;
        case 2: x = p.W - 1 - i; y = c; break;
        default: x = c; y = p.H - 1 - i; break;
    }
}

__device__ __forceinline__ bool survives(const DevState& s, int j, float sv)
{
    return sv > s.mie_prev_score[j] && sv >= s.mie_smp_score[j];
}

__global__ void k_mie_prepare(DevParams p, DevState s)
{
    __shared__ FramesF f;
    load_frames32(p, s, f);
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= p.N) return;
    const int k = *s.iter;
    const int x = j % p.W, y = j / p.W;
    const U64x4 r = philox4x64_10((uint64_t)j, 0ull, (uint64_t)k, (uint64_t)kStreamDepth, p.seed, p.window_id);
    const float u = (float)(r.v[0] >> 40) * (1.f / 16777216.f);
    const float smp = 1.f / fmaf(u, p.inv_depth_max - p.inv_depth_min, p.inv_depth_min);
    const float prev = mie_score(p, s, f, x, y, s.theta[j]);
    s.mie_prev_score[j] = prev;
    s.mie_smp[j] = smp;
    s.mie_smp_score[j] = mie_score_above(p, s, f, x, y, smp, prev);   // below S(prev) its value has no effect
}

// own value of pixel j (before the sweep overwrites theta)
__device__ __forceinline__ float own_value(const DevState& s, int j)
{
    return s.mie_smp_score[j] > s.mie_prev_score[j] ? s.mie_smp[j] : s.theta[j];
}

__global__ void k_mie_runs(DevParams p, DevState s)
{
    __shared__ FramesF f;
    load_frames32(p, s, f);
    const int dir = (*s.iter) & 3;
    const bool rows = (dir == 0 || dir == 2);
    const int len = rows ? p.W : p.H;
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= p.N) return;
    const int c = id / len, i = id % len;
    int x, y;
    chain_xy(p, dir, c, i, x, y);
    const int j = y * p.W + x;
    const float v = own_value(s, j);
    int e = i + 1;
    int steps = 0;
    while (e < len && steps < kRunCap) {
        int xe, ye;
        chain_xy(p, dir, c, e, xe, ye);
        if (!survives(s, ye * p.W + xe, mie_score(p, s, f, xe, ye, v))) break;
        ++e;
        ++steps;
    }
    s.mie_next[j] = (steps == kRunCap && e < len) ? -e : e;
}

constexpr int kResolveWarps = 16, kResolveThreads = 32 * kResolveWarps;
constexpr int kMaxChain = kMaxImageSide;

// A warp tests 32 >> lg positions of a chain at a time, 2^lg lanes to a position, a frame each
// (two from T = 9 on); the frames' terms are independent, only their sum is in order.
__device__ __forceinline__ int test_lanes_log2(const DevParams& p) { return p.T > 4 ? 3 : (p.T > 2 ? 2 : p.T - 1); }

// The first of the positions pos, pos + 1, ... of chain c at which the warp finds v lost, or
// pos + (32 >> lg) if it survives them all. Positions past the chain's end are lost.
__device__ int mie_test(const DevParams& p, const DevState& s, const FramesF& f, int dir, int c, int len, int pos, int lg, float v)
{
    const int lane = threadIdx.x & 31, mask = (1 << lg) - 1, sub = lane & mask, first = lane - sub, q = pos + (lane >> lg);
    int x, y;
    chain_xy(p, dir, c, min(q, len - 1), x, y);
    const int j = y * p.W + x;
    float term[2] = {0.f, 0.f};
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int t = (u << lg) + sub + 1;
        if (t <= p.T) term[u] = __fmul_rn(s.qs[(size_t)(t - 1) * p.N + j], depth_ell_fast(p, f.v[t - 1], s.flows, t, x, y, v));
    }
    float acc = 0.f;
    for (int t = 0; t < p.T; ++t) acc = __fadd_rn(acc, __shfl_sync(0xffffffffu, t <= mask ? term[0] : term[1], first + (t & mask)));
    const unsigned lost = __ballot_sync(0xffffffffu, q >= len || !survives(s, j, nan_to_ninf(acc)));
    return pos + (lost ? (__ffs(lost) - 1) >> lg : 32 >> lg);
}

// End of the run of v, which survived up to position `pos` of chain c, by one warp; -q if
// it is alive at a position q >= limit, not tested yet.
__device__ int mie_run_end(const DevParams& p, const DevState& s, const FramesF& f, int dir, int c, int len, int pos, int limit, int lg,
                           float v)
{
    for (;;) {
        const int end = pos + (32 >> lg);
        pos = mie_test(p, s, f, dir, c, len, pos, lg, v);
        if (pos < end) return min(pos, len);
        if (pos >= limit) return pos < len ? -pos : len;
    }
}

// Resolution of one chain per block. The walk r -> end of r's run depends on nothing
// but r, so walks from different positions join at the first reset they share. Each
// warp first walks its own part of the chain from the part's first position, and
// whatever a run that reached the cap costs is paid by the warps side by side; then
// warp 0 follows the true walk from one part to the next, step by step until it meets
// the part's own walk, from there on by its result. A chain's runs one after another,
// tested by the whole block, took 212 us at 1242 x 375, T = 8 with a cap of 8; the parts
// take 65 with that cap and 89 with 2 (see kRunCap). With 8 or 32 parts instead of 16 a
// first version took 101 and 146 us where it took 108.
//
// A run that goes on kOver positions past its warp's part is left open: the true walk may
// never come by it, and where it does (or meets a run of its own that outlives kAlone
// positions) the whole block tests the next positions at once. Followed to their ends by
// the parts' warps, runs of hundreds of positions, as over a plane whose depth was poor
// and whose flows are quiet, made a sweep 958 us at 1242 x 375, T = 8; now 396, with
// every test by the block (before there were parts) 545. With short runs 250 us along
// rows and 291 along columns (266 and 388). The lanes' shares are shifts and masks: with
// divisions by the lanes per position a sweep took 9 % longer. Tried: all warps walking
// (3 % longer on short runs), long runs a lane per position instead of a frame per lane
// (no change), two blocks per SM instead of three (56 registers instead of 40 and a few
// spills: 2 % longer at this size, 4 % shorter at 320 x 240).
constexpr int kOver = 32, kAlone = 16;

__global__ void __launch_bounds__(kResolveThreads, 3) k_mie_resolve(DevParams p, DevState s)
{
    __shared__ FramesF f;
    __shared__ short origin[kMaxChain];
    __shared__ int next_s[kMaxChain];
    __shared__ float own_s[kMaxChain];
    __shared__ unsigned char reset[kMaxChain];             // 1: on the part's own walk, 2: on the true one before they meet
    __shared__ int part_end[kResolveWarps], part_last[kResolveWarps], part_from[kResolveWarps], last_s[kResolveWarps];
    __shared__ int first_lost[3];
    load_frames32(p, s, f);
    const int dir = (*s.iter) & 3;
    const bool rows = (dir == 0 || dir == 2);
    const int n_chains = rows ? p.H : p.W;
    const int len = rows ? p.W : p.H;
    const int c = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (c >= n_chains) return;
    for (int q = threadIdx.x; q < len; q += kResolveThreads) {
        int x, y;
        chain_xy(p, dir, c, q, x, y);
        next_s[q] = s.mie_next[y * p.W + x];
        own_s[q] = own_value(s, y * p.W + x);
        reset[q] = 0;
    }
    __syncthreads();
    const int part = (len + kResolveWarps - 1) / kResolveWarps, lg = test_lanes_log2(p);
    {
        const int stop = min((warp + 1) * part, len);
        int r = min(warp * part, len), last = 0;
        while (r >= 0 && r < stop) {
            last = r;
            int e = next_s[r];
            if (e < 0) {
                e = mie_run_end(p, s, f, dir, c, len, -e, stop + kOver, lg, own_s[r]);
                __syncwarp();
                if (lane == 0) next_s[r] = e;
            }
            if (lane == 0) reset[r] = 1;
            r = e;
        }
        if (lane == 0) {
            part_end[warp] = r;
            part_last[warp] = last;
        }
    }
    if (threadIdx.x == 0) first_lost[0] = kMaxChain;
    __syncthreads();
    // warp 0 walks until it meets an open run that it leaves to the block, or the chain's end
    __shared__ int open_pos;
    __shared__ float open_v;
    const int wide = 32 >> lg;
    int r = 0, k = 0, step = 0;
    for (;;) {
        if (warp == 0) {
            int pos = 0;
            float v = 0.f;
            while (k < kResolveWarps) {
                if (r >= min((k + 1) * part, len)) {         // the walk passes the part by
                    if (lane == 0) part_from[k] = len;
                    ++k;
                    continue;
                }
                int e;
                if (reset[r] == 1) {                          // it goes on as the part's own
                    if (lane == 0) part_from[k] = r;
                    e = part_end[k];
                    v = own_s[part_last[k]];
                    ++k;
                } else {
                    if (lane == 0) reset[r] = 2;
                    e = next_s[r];
                    v = own_s[r];
                }
                if (e < 0) e = mie_run_end(p, s, f, dir, c, len, -e, kAlone - e, lg, v);
                if (e < 0) {
                    pos = -e;
                    break;
                }
                r = e;
            }
            if (lane == 0) {
                open_pos = pos;
                open_v = v;
            }
        }
        __syncthreads();
        int pos = open_pos;
        if (pos == 0) break;
        const float v = open_v;
        // the run's end, tested by the whole block
        for (;; pos += wide * kResolveWarps) {
            const int mine = pos + warp * wide, slot = step % 3;
            const int end = mie_test(p, s, f, dir, c, len, mine, lg, v);
            step += 1;
            if (lane == 0 && end < mine + wide) atomicMin(&first_lost[slot], end);
            if (threadIdx.x == 0) first_lost[step % 3] = kMaxChain;     // read for the last time two steps ago
            __syncthreads();
            const int at = first_lost[slot];
            r = min(at, len);
            if (at < kMaxChain || pos + wide * kResolveWarps >= len) break;
        }
    }
    __syncthreads();
    // origin of each position: the last reset of the true walk up to it, a contiguous
    // piece per thread, then a scan over the pieces
    const int per = (len + kResolveThreads - 1) / kResolveThreads, q0 = threadIdx.x * per, q1 = min(q0 + per, len);
    auto is_reset = [&](int q) { return reset[q] == 2 || (reset[q] == 1 && q >= part_from[q / part]); };
    int last = -1;
    for (int q = q0; q < q1; ++q)
        if (is_reset(q)) last = q;
    int before = last;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, before, o);
        if (lane >= o) before = max(before, v);
    }
    if (lane == 31) last_s[warp] = before;
    before = __shfl_up_sync(0xffffffffu, before, 1);
    if (lane == 0) before = -1;
    __syncthreads();
    for (int w = 0; w < warp; ++w) before = max(before, last_s[w]);
    for (int q = q0; q < q1; ++q) {
        if (is_reset(q)) before = q;
        origin[q] = (short)before;
    }
    __syncthreads();
    // new depths and labels (the chain's own values are in shared memory)
    for (int q = threadIdx.x; q < len; q += kResolveThreads) {
        int x, y;
        chain_xy(p, dir, c, q, x, y);
        const int j = y * p.W + x;
        s.theta[j] = own_s[origin[q]];
        s.labels[j] = origin[q] != q ? 1 : (s.mie_smp_score[j] > s.mie_prev_score[j] ? 2 : 0);
    }
}

void launch_mie(const DevParams& p, const DevState& s, cudaStream_t st)
{
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    k_mie_prepare<<<nb, kPixThreads, 0, st>>>(p, s);
    k_mie_runs<<<nb, kPixThreads, 0, st>>>(p, s);
    k_mie_resolve<<<p.H > p.W ? p.H : p.W, kResolveThreads, 0, st>>>(p, s);
}

// ---------------------------------------------------------------------------
// Iteration counter.
// ---------------------------------------------------------------------------
__global__ void k_set_iter(int* iter, int k) { *iter = k; }
__global__ void k_advance_iter(int* iter) { *iter += 1; }

void launch_set_iteration(const DevState& s, int k, cudaStream_t st) { k_set_iter<<<1, 1, 0, st>>>(s.iter, k); }
void launch_advance_iteration(const DevState& s, cudaStream_t st) { k_advance_iter<<<1, 1, 0, st>>>(s.iter); }

}  // namespace vd
