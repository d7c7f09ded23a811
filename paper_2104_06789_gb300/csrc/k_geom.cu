// FP64-geometry passes of the VOLDOR loop: pose preparation (the dense
// scoring's per-pixel records), the E-step emissions (also the unsmoothed
// rigidness update) and forward-backward smoothing of the rigidness.
//
// Geometry is FP64 and likelihood arithmetic FP32 (k_prep_count/k_prep_write,
// k_emissions, neg_ell). Unlike the MIE sweep's translation unit this one is
// compiled with FMA contraction: none of its results is compared bit for bit
// with another kernel's, and fused FP64 multiply-adds cut the FP64
// instructions of the geometry (this GPU's FP64 rate is a small fraction of
// its FP32 rate).
#include <algorithm>

#include "df32.cuh"
#include "score_ops.cuh"
#include "voldor_internal.cuh"

namespace vd {

// ---------------------------------------------------------------------------
// Pose preparation of frame t: one record per pixel whose pi_{t-1} is valid,
// compacted in pixel order. Both passes compute each pixel's point in camera
// t-1, P = C_{t-1} theta K^-1 [x y 1], and pi_{t-1} in df32 (float-float on
// the FP32 pipe, ~44 bits: the validity test 0 <= pi_{t-1} <= size - 1 and
// the bilinear sample position are those of an FP64 computation but within
// ~1e-11 px). The count pass counts the valid pixels per block and stores
// per-warp ballots of them, and its last block to finish scans the counts
// into block offsets; the write pass recomputes the same values, samples the
// flow at pi_{t-1} bilinearly (df32) and writes the records at its block's
// offset.
// ---------------------------------------------------------------------------
struct PrepGeo {
    DF Px, Py, Pz, iz, u, v;       // iz = 1 / Pz (set for t > 1 where Pz > 0)
    bool valid;
};

// C_{t-1} as float-float pairs, written by the frame set-up
__device__ __forceinline__ void load_cum_df(const DevState& s, int t, DF* C)
{
    if (threadIdx.x < 12) {
        const float* c = s.cum_df + 24 * (t - 1) + 2 * threadIdx.x;
        C[threadIdx.x] = DF{c[0], c[1]};
    }
    __syncthreads();
}

__device__ __forceinline__ PrepGeo prep_geometry(const DevParams& p, const DF* C, int t, int j, float th)
{
    int x, y;
    pixel_xy(p, j, x, y);
    const DF fx{p.kdf[0], p.kdf[1]}, fy{p.kdf[2], p.kdf[3]}, cx{p.kdf[4], p.kdf[5]}, cy{p.kdf[6], p.kdf[7]};
    const DF ifx{p.kdf[8], p.kdf[9]}, ify{p.kdf[10], p.kdf[11]};
    PrepGeo g;
    const float xf = small_int_to_float(x), yf = small_int_to_float(y);
    const DF X = df_mul(df_mul(df_add(df_neg(cx), xf), ifx), th);
    const DF Y = df_mul(df_mul(df_add(df_neg(cy), yf), ify), th);
    const DF Z = df_of(th);
    g.u = df_of(xf);
    g.v = df_of(yf);
    if (t == 1) {
        g.Px = X; g.Py = Y; g.Pz = Z;
    } else {
        g.Px = df_add(df_add(df_mul(C[0], X), df_mul(C[1], Y)), df_add(df_mul(C[2], Z), C[3]));
        g.Py = df_add(df_add(df_mul(C[4], X), df_mul(C[5], Y)), df_add(df_mul(C[6], Z), C[7]));
        g.Pz = df_add(df_add(df_mul(C[8], X), df_mul(C[9], Y)), df_add(df_mul(C[10], Z), C[11]));
    }
    g.valid = df_gt0(g.Pz);
    if (g.valid && t > 1) {
        g.iz = df_div(df_of(1.f), g.Pz);
        g.u = df_add(df_mul(df_mul(fx, g.Px), g.iz), cx);
        g.v = df_add(df_mul(df_mul(fy, g.Py), g.iz), cy);
    }
    g.valid = g.valid && df_ge(g.u, 0.f) && df_le(g.u, small_int_to_float(p.W - 1)) && df_ge(g.v, 0.f) &&
              df_le(g.v, small_int_to_float(p.H - 1));
    return g;
}

// True if the pose M (hi parts of T_t) leaves a smaller residual at a valid pixel than no
// motion at all, with the pixel's own flow f instead of the one at its projection (FP32).
// The scoring's operands are formed around a reference pose that every hypothesis is the
// difference from; around one far from the hypotheses the differences cancel against it
// and the scores lose their digits (a translation of 70 in a scene 2 to 20 deep cost
// 1.2e-5 of them, one of 2e5 cost 7 %). So the current pose is the reference only where
// it explains more of the pixels than the identity does, whose part of a residual is the
// flow itself. The vote takes 0.5 to 1 us of the count; in a kernel of its own, beside P3P,
// it took one block 8 us, and score_hypotheses, which has no P3P, 10 us a call.
__device__ __forceinline__ bool pose_explains(const DevParams& p, const float* M, const PrepGeo& g, float2 f)
{
    const float iz = 1.f / g.Pz.hi, x = g.Px.hi * iz, y = g.Py.hi * iz;
    const float fu = f.x * p.inv_fx, fv = f.y * p.inv_fy;
    const float ax = fmaf(M[0] - 1.f, x, fmaf(M[1], y, fmaf(M[3], iz, M[2])));
    const float ay = fmaf(M[4], x, fmaf(M[5] - 1.f, y, fmaf(M[7], iz, M[6])));
    const float az = fmaf(M[8], x, fmaf(M[9], y, fmaf(M[11], iz, M[10] - 1.f))), den = 1.f + az;
    const float U = fmaf(x + fu, az, fu - ax), V = fmaf(y + fv, az, fv - ay);
    return den > 0.f && fabsf(U) + fabsf(V) <= (fabsf(fu) + fabsf(fv)) * den;
}

__global__ void __launch_bounds__(kPixThreads) k_prep_count(DevParams p, DevState s, int t)
{
    __shared__ DF C[12];
    __shared__ float M[12];
    __shared__ int votes_s, votes_all;
    const int j = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // one warp of a block votes on the reference pose, another one in each block
    const bool voter = warp == (blockIdx.x & (kPixThreads / 32 - 1));
    float2 f = make_float2(0.f, 0.f);
    if (voter && j < p.N) f = load_flow(s.flows, p.flow_f16, (size_t)(t - 1) * p.N + j);
    if (threadIdx.x >= 32 && threadIdx.x < 44) M[threadIdx.x - 32] = s.poses_df[24 * (t - 1) + 2 * (threadIdx.x - 32)];
    load_cum_df(s, t, C);
    PrepGeo g;
    g.valid = false;
    if (j < p.N) g = prep_geometry(p, C, t, j, s.theta[j]);
    const bool valid = g.valid;
    // per-warp ballots of the valid pixels: with the block offsets they map
    // the i-th valid pixel (pixel order) to its index for the minimal groups
    const unsigned bal = __ballot_sync(0xffffffffu, valid);
    if (lane == 0) s.pix_vmask[j >> 5] = bal;
    if (voter) {
        const int votes = __popc(__ballot_sync(0xffffffffu, valid && pose_explains(p, M, g, f)));
        if (lane == 0) votes_s = (2 * votes - __popc(bal)) * 65536;
    }
    if (threadIdx.x == 0) votes_all = 0;
    const int cnt = __syncthreads_count(valid);
    // the last block to finish turns the block counts into block offsets
    // (exclusive scan, in place), sets the record count and clears the P3P
    // claim counters and coarse counts of the frame; no block waits
    __shared__ bool last;
    if (threadIdx.x == 0) {
        s.pix_block_count[blockIdx.x] = cnt + votes_s;       // above the count: the votes for less those against
        __threadfence();
        last = atomicAdd(s.prep_done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int nb = gridDim.x, per = (nb + blockDim.x - 1) / blockDim.x;
    const int b0 = min((int)threadIdx.x * per, nb), b1 = min(b0 + per, nb);
    volatile int* counts = s.pix_block_count;
    int local = 0, votes = 0;
    for (int b = b0; b < b1; ++b) {
        const int c = counts[b];
        local += c & 0xffff;
        votes += c >> 16;
    }
    votes = __reduce_add_sync(0xffffffffu, votes);
    if (lane == 0) atomicAdd(&votes_all, votes);
    __shared__ int wsum[kPixThreads / 32];
    int incl = local;
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    int off = before + incl - local;
    for (int b = b0; b < b1; ++b) {
        const int c = counts[b] & 0xffff;
        counts[b] = off;
        off += c;
    }
    static_assert(kP3PMaxBlocks <= kPixThreads, "one count a thread");
    if (threadIdx.x < kP3PMaxBlocks) s.block_sols[threadIdx.x] = 0;
    if (threadIdx.x == blockDim.x - 1) {
        *s.pix_count = off;
        *s.prep_done = 0u;
        *s.p3p_claims = 0;
        *s.p3p_done = 0ull;
        *s.sc_wild = 0;
        *s.sc_ref = votes_all >= 0;
    }
}

// What bounds the write: float-float arithmetic at three quarters of the issue slots; it
// leaves 212 bytes a pixel for the scoring (21 us at 640 x 480). The two residual models
// apart: with the choice at run time the kernel needs 62 registers instead of 40, and
// the P3P beside it starts later (50 to 65 us a frame at 640 x 480).
template <bool kGauss>
__global__ void __launch_bounds__(kPixThreads) k_prep_write(DevParams p, DevState s, int t)
{
    __shared__ DF C[12], T0[12];
    __shared__ int warp_sum[kPixThreads / 32];
    if (threadIdx.x < 12) {                               // the reference pose (pose_explains)
        const float* c = s.poses_df + 24 * (t - 1) + 2 * threadIdx.x;
        const float hi = c[0], lo = c[1];
        const bool current = *s.sc_ref != 0;
        T0[threadIdx.x] = DF{current ? hi : (threadIdx.x % 5 == 0 ? 1.f : 0.f), current ? lo : 0.f};
    }
    load_cum_df(s, t, C);
    const int base = s.pix_block_count[blockIdx.x];      // this block's offset (set by the count pass)
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const size_t N = (size_t)p.N;
    PrepGeo g;
    g.valid = false;
    if (j < p.N) g = prep_geometry(p, C, t, j, s.theta[j]);
    const unsigned bal = __ballot_sync(0xffffffffu, g.valid);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_sum[warp] = __popc(bal);
    __syncthreads();
    int rank = __popc(bal & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) rank += warp_sum[w];
    if (g.valid) {
        const int x0 = min(df_floor(g.u), p.W - 2), y0 = min(df_floor(g.v), p.H - 2);
        const DF ax = df_add(g.u, -small_int_to_float(x0)), ay = df_add(g.v, -small_int_to_float(y0));
        const size_t fb = (size_t)(t - 1) * N + (size_t)y0 * p.W + x0;
        const float2 f00 = load_flow(s.flows, p.flow_f16, fb), f10 = load_flow(s.flows, p.flow_f16, fb + 1);
        const float2 f01 = load_flow(s.flows, p.flow_f16, fb + p.W);
        const float2 f11 = load_flow(s.flows, p.flow_f16, fb + p.W + 1);
        const DF gu0 = df_add(df_mul(df_two_sum(f10.x, -f00.x), ax), f00.x);
        const DF gu1 = df_add(df_mul(df_two_sum(f11.x, -f01.x), ax), f01.x);
        const DF gv0 = df_add(df_mul(df_two_sum(f10.y, -f00.y), ax), f00.y);
        const DF gv1 = df_add(df_mul(df_two_sum(f11.y, -f01.y), ax), f01.y);
        const DF fud = df_add(gu0, df_mul(df_sub(gu1, gu0), ay));
        const DF fvd = df_add(gv0, df_mul(df_sub(gv1, gv0), ay));
        const DF ifx{p.kdf[8], p.kdf[9]};
        const float fu = df_to_float(fud), fv = df_to_float(fvd);
        const DF ut = df_mul(fud, ifx), vt = df_mul(fvd, ifx);
        const DF iz = t == 1 ? df_div(df_of(1.f), g.Pz) : g.iz;
        const float n = sqrtf(fmaf(fu, fu, fv * fv));
        const float fx2 = df_to_float(df_mul(DF{p.kdf[0], p.kdf[1]}, DF{p.kdf[0], p.kdf[1]}));
        // features of the projection (score_ops.cuh), in float-float
        const DF xn = df_mul(g.Px, iz), yu = df_mul(g.Py, iz), yn = df_mul(yu, p.fy_over_fx);
        const DF X = df_add(xn, ut), Y = df_add(yn, vt);
        // a = (T - I) p at the reference pose T: a_z0, U0 = X a_z0 - a_x0 + ut, V0 alike
        auto row = [&](int r) {
            const DF e0 = r == 0 ? df_add(T0[0], -1.f) : T0[4 * r], e1 = r == 1 ? df_add(T0[5], -1.f) : T0[4 * r + 1];
            const DF e2 = r == 2 ? df_add(T0[10], -1.f) : T0[4 * r + 2];
            return df_add(df_add(df_mul(e0, xn), df_mul(e1, yu)), df_add(e2, df_mul(T0[4 * r + 3], iz)));
        };
        const DF az0 = row(2);
        const DF U0 = df_add(df_sub(df_mul(X, az0), row(0)), ut);
        const DF V0 = df_add(df_sub(df_mul(Y, az0), df_mul(row(1), p.fy_over_fx)), vt);
        __align__(16) __nv_bfloat16 o[kScPixCols];
        const DF up{1.f, (float)(kScUntruncate - 1.0)};
        const Slice3 fs[3] = {slice3(xn), slice3(yn), slice3(iz)};
        pixel_block_s(fs, slice3(df_mul(az0, up)), o);
        // under the Gaussian model the scoring adds the references itself, up to what FP32 leaves of them
        const Slice3 fu4[4] = {slice3(df_mul(X, xn)), slice3(df_mul(X, yn)), slice3(df_mul(X, iz)), slice3(X)};
        pixel_block_x(fu4, kGauss ? slice3(U0.lo, 0.f) : slice3(df_mul(U0, up)), fs, o + 32);
        const Slice3 fv4[4] = {slice3(df_mul(Y, xn)), slice3(df_mul(Y, yn)), slice3(df_mul(Y, iz)), slice3(Y)};
        pixel_block_x(fv4, kGauss ? slice3(V0.lo, 0.f) : slice3(df_mul(V0, up)), fs, o + 64);
        const int i = base + rank;
        unsigned char* d = s.sc_pix + (size_t)(i / kScTilePix) * kScTileBytes + ((i % kScTilePix) / 8) * 128 + (i % 8) * 16;
#pragma unroll
        for (int q = 0; q < kScPixCols / 8; ++q)
            *reinterpret_cast<uint4*>(d + q * (kScTilePix * 16)) = *reinterpret_cast<const uint4*>(o + 8 * q);
        float4 cst;
        if (kGauss) {
            const GaussConst gc = gauss_const(p, n);
            cst = make_float4(fx2 * gc.inv_alpha, -gc.x_mu * gc.inv_alpha, U0.hi, 0.f);
            s.sc_xmu[i] = V0.hi;
        } else {
            const FiskConst fc = fisk_const(p, n);
            cst = make_float4(fc.beta, fc.beta * (p.log2_fx2 - fc.log2_alpha), fx2 * fc.mu_over_beta, 0.f);
            // At x_mu, where a pixel behind the camera is taken, r = Cp xs (2^s + 2 + 2^-s) is 1; with
            // |s| beyond 128 (flows of thousands of pixels with a shape that is not small) its
            // factors overflow. Only one power of two counts there: s is moved to 80.
            if (fabsf(fc.s_mu) > 100.f) {
                cst.y = copysignf(80.f, fc.s_mu) - fc.beta * (log2f(fc.x_mu) - p.log2_fx2);
                cst.z = fx2 * 0x1p-80f / fc.x_mu;
            }
            s.sc_xmu[i] = fc.x_mu / fx2;
        }
        cst.w = s.wmap[(size_t)(t - 1) * N + j];
        s.sc_cst[i] = cst;
        if (!(fabsf(xn.hi) < kScWild && fabsf(yn.hi) < kScWild && fabsf(iz.hi) < kScWild)) atomicOr(s.sc_wild, 1);
    }
}

void launch_prep_count(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    k_prep_count<<<nb, kPixThreads, 0, st>>>(p, s, t);
}

void launch_prep_write(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    if (p.residual == VOLDOR_RESIDUAL_GAUSSIAN) k_prep_write<true><<<nb, kPixThreads, 0, st>>>(p, s, t);
    else k_prep_write<false><<<nb, kPixThreads, 0, st>>>(p, s, t);
}

void launch_pose_prep(const DevParams& p, const DevState& s, int t, cudaStream_t st)
{
    launch_prep_count(p, s, t, st);
    launch_prep_write(p, s, t, st);
}

// Emissions rho/(rho+mu) of every (t, j) at the current depth (E-step input)
// or, written into W, the unsmoothed rigidness update: per (t, j) the rigid
// flow and residual in df32 (float-float, on the FP32 pipe) and the
// likelihood in FP32 (neg_ell); log(1/2) where the model takes rho := mu
// (pi_{t-1} invalid or the point behind camera t). The point is carried from
// frame to frame: the point in camera t (T_t applied to the point in camera
// t-1) and its projection pi_t are the next frame's point in camera (t+1)-1
// and pi_{(t+1)-1}, since C_t X = T_t (C_{t-1} X), so each frame transforms
// and projects once (the frame set-up's float-float copy of T_t). The residual xi - v_ob (tenths of a pixel) is the
// difference of quantities of up to hundreds of pixels: the sample position,
// the bilinear flow (in lerp form, with df32 fractions) and the rigid flow
// are all kept in df32 and only the residual is rounded to FP32.
__global__ void __launch_bounds__(kPixThreads) k_emissions(DevParams p, DevState s, float* out)
{
    __shared__ DF Tdf[kMaxT][12];
    for (int i = threadIdx.x; i < p.T * 12; i += blockDim.x)
        Tdf[i / 12][i % 12] = DF{s.poses_df[2 * i], s.poses_df[2 * i + 1]};
    __syncthreads();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= p.N) return;
    int x, y;
    pixel_xy(p, j, x, y);
    const DF fx{p.kdf[0], p.kdf[1]}, fy{p.kdf[2], p.kdf[3]}, cx{p.kdf[4], p.kdf[5]}, cy{p.kdf[6], p.kdf[7]};
    const DF ifx{p.kdf[8], p.kdf[9]}, ify{p.kdf[10], p.kdf[11]};
    const float th = s.theta[j];
    // the point in camera t-1 (camera 0 for t = 1) and pi_{t-1}
    const float xf = small_int_to_float(x), yf = small_int_to_float(y);
    DF Px = df_mul(df_mul(df_add(df_neg(cx), xf), ifx), th);
    DF Py = df_mul(df_mul(df_add(df_neg(cy), yf), ify), th);
    DF Pz = df_of(th);
    DF u = df_of(xf), v = df_of(yf);
    bool front = th > 0.f;                          // P_z > 0 and (u, v) defined
    const float Wm1 = small_int_to_float(p.W - 1), Hm1 = small_int_to_float(p.H - 1);
    for (int t = 1; t <= p.T; ++t) {
        float ell = -0.69314718055994531f;          // rho := mu
        DF fu = df_of(0.f), fv = df_of(0.f);
        const bool valid_prev = front && df_ge(u, 0.f) && df_le(u, Wm1) && df_ge(v, 0.f) && df_le(v, Hm1);
        if (valid_prev) {
            const int x0 = min(df_floor(u), p.W - 2), y0 = min(df_floor(v), p.H - 2);
            const DF ax = df_add(u, -small_int_to_float(x0)), ay = df_add(v, -small_int_to_float(y0));
            const size_t base = (size_t)(t - 1) * p.N + (size_t)y0 * p.W + x0;
            const float2 f00 = load_flow(s.flows, p.flow_f16, base), f10 = load_flow(s.flows, p.flow_f16, base + 1);
            const float2 f01 = load_flow(s.flows, p.flow_f16, base + p.W);
            const float2 f11 = load_flow(s.flows, p.flow_f16, base + p.W + 1);
            // f00 + ax (f10 - f00), f01 + ax (f11 - f01), then the same in y
            const DF gu0 = df_add(df_mul(df_two_sum(f10.x, -f00.x), ax), f00.x);
            const DF gu1 = df_add(df_mul(df_two_sum(f11.x, -f01.x), ax), f01.x);
            const DF gv0 = df_add(df_mul(df_two_sum(f10.y, -f00.y), ax), f00.y);
            const DF gv1 = df_add(df_mul(df_two_sum(f11.y, -f01.y), ax), f01.y);
            fu = df_add(gu0, df_mul(df_sub(gu1, gu0), ay));
            fv = df_add(gv0, df_mul(df_sub(gv1, gv0), ay));
        }
        const DF* Tt = Tdf[t - 1];
        const DF Qx = df_add(df_add(df_mul(Tt[0], Px), df_mul(Tt[1], Py)), df_add(df_mul(Tt[2], Pz), Tt[3]));
        const DF Qy = df_add(df_add(df_mul(Tt[4], Px), df_mul(Tt[5], Py)), df_add(df_mul(Tt[6], Pz), Tt[7]));
        const DF Qz = df_add(df_add(df_mul(Tt[8], Px), df_mul(Tt[9], Py)), df_add(df_mul(Tt[10], Pz), Tt[11]));
        const bool front_t = df_gt0(Qz);
        DF uq = df_of(0.f), vq = df_of(0.f);
        if (front_t) {
            const DF iq = df_div(df_of(1.f), Qz);
            uq = df_add(df_mul(df_mul(fx, Qx), iq), cx);
            vq = df_add(df_mul(df_mul(fy, Qy), iq), cy);
        }
        if (valid_prev && front_t) {
            const float ru = df_to_float(df_sub(df_sub(uq, u), fu));
            const float rv = df_to_float(df_sub(df_sub(vq, v), fv));
            const float xs = fminf(fmaxf(fmaf(ru, ru, rv * rv), p.x_min), p.x_max);
            const float fuf = df_to_float(fu), fvf = df_to_float(fv);
            ell = -neg_ell(p, xs, sqrtf(fmaf(fuf, fuf, fvf * fvf)), false);
        }
        out[(size_t)(t - 1) * p.N + j] = expf(ell);
        Px = Qx; Py = Qy; Pz = Qz;
        u = uq; v = vq;
        front = front_t;
    }
}

void launch_emissions(const DevParams& p, const DevState& s, float* out, cudaStream_t st)
{
    const int nb = (p.N + kPixThreads - 1) / kPixThreads;
    k_emissions<<<nb, kPixThreads, 0, st>>>(p, s, out);
}

// ---------------------------------------------------------------------------
// Forward-backward (Eqs. 12-14) on every chain of every frame, one warp per
// chain. Emissions (1 - w, w) are read from s.qs and replaced by the
// smoothed q(W = 1). With A = [[g, h], [h, g]] (g = gamma, h = 1 - gamma):
//   forward   f_0 = e_0,  f_i = diag(e_i) A f_{i-1}
//   backward  b_{n-1} = 1, b_i = A diag(e_{i+1}) b_{i+1}
//   q_i = f_i .* b_i (normalised),
// every message renormalised at every step. The chain is cut into 32
// contiguous segments, one per lane; each lane forms the product of its
// segment's 2x2 transfer matrices (renormalised by their entry sum, all
// entries are non-negative), a 5-step shuffle scan gives each lane the
// product of the segments before it (forward) or after it (backward), and
// each lane then walks its own segment with the step-by-step recursion from
// the message entering it.
//
// A block stages neighbouring chains in shared memory, emissions and forward messages,
// and moves them between there and global memory in whole rows (or, along columns, some
// columns of a row at a time): kFbChains of the longer direction's chains, and of the
// shorter ones what fits in the same room, up to a chain per warp. With the lanes'
// strided accesses in global memory the kernel took 107 us at 1242 x 375, T = 8; now
// 66 (58 along rows, 74 along columns; 90 with four chains there too). What bounds it
// now: the latency of a step (up to two divisions) times four passes over a segment,
// with the chains an SM has room for.
// ---------------------------------------------------------------------------
constexpr int kFbChains = 4, kFbMaxWarps = 32;

// Floats of a chain's row in shared memory: 32 segments, padded to an odd length so
// that the lanes' steps fall into different banks.
__host__ __device__ constexpr int fb_segment(int len) { return (len + 31) / 32; }
__host__ __device__ constexpr int fb_row(int len) { return 32 * (fb_segment(len) | 1); }

// Warps of a block: 8, but of a strip whose longer chains leave an SM room for two blocks or
// one, as many as the shorter chains fill (4096 x 16, T = 8, columns: 77 us, 136 with 8).
__host__ inline int fb_warps(int most, int least)
{
    const int room = 227 * 1024 / (kFbChains * 3 * fb_row(most) * (int)sizeof(float));
    const int fit = kFbChains * fb_row(most) / fb_row(least);
    return room > 2 ? 8 : std::max(8, std::min(fit, kFbMaxWarps / room));
}

// Chains of length len to a block of `warps` whose room is kFbChains chains of length most.
__host__ __device__ inline int fb_chains(int len, int most, int warps)
{
    const int fit = kFbChains * fb_row(most) / fb_row(len);
    return fit < warps ? fit : warps;
}

struct M22 {
    float a, b, c, d;   // [[a, b], [c, d]]
};

__device__ __forceinline__ M22 m22_mul(const M22& x, const M22& y)
{
    M22 r{x.a * y.a + x.b * y.c, x.a * y.b + x.b * y.d, x.c * y.a + x.d * y.c, x.c * y.b + x.d * y.d};
    const float s = r.a + r.b + r.c + r.d;
    if (s > 0.f) {
        const float is = 1.f / s;
        r.a *= is; r.b *= is; r.c *= is; r.d *= is;
    }
    return r;
}

__device__ __forceinline__ M22 m22_shfl(const M22& x, int src_delta, bool up)
{
    M22 r;
    if (up) {
        r.a = __shfl_up_sync(0xffffffffu, x.a, src_delta); r.b = __shfl_up_sync(0xffffffffu, x.b, src_delta);
        r.c = __shfl_up_sync(0xffffffffu, x.c, src_delta); r.d = __shfl_up_sync(0xffffffffu, x.d, src_delta);
    } else {
        r.a = __shfl_down_sync(0xffffffffu, x.a, src_delta); r.b = __shfl_down_sync(0xffffffffu, x.b, src_delta);
        r.c = __shfl_down_sync(0xffffffffu, x.c, src_delta); r.d = __shfl_down_sync(0xffffffffu, x.d, src_delta);
    }
    return r;
}

// One chain by a warp: its emissions in shared memory are replaced by q. e, fw: the
// lane's segment (e[LP] is the next lane's first element).
__device__ __forceinline__ void fb_chain(const DevParams& p, int len, float* e, float2* fw, const float* chain)
{
    const int lane = threadIdx.x & 31;
    const float g = p.gamma, h = 1.f - p.gamma;
    const int L = fb_segment(len), LP = L | 1;
    const int i0 = min(lane * L, len), i1 = min(i0 + L, len);    // this lane's segment [i0, i1)
    const bool has = i0 < i1;

    // ---- forward: segment products of diag(e_i) A for i in [max(i0, 1), i1)
    M22 P{1.f, 0.f, 0.f, 1.f};
    for (int i = (i0 > 0 ? i0 : 1); i < i1; ++i) {
        const float w = e[i - i0];
        const M22 Mi{(1.f - w) * g, (1.f - w) * h, w * h, w * g};
        P = m22_mul(Mi, P);
    }
    // inclusive scan: S_k = P_k ... P_0 (later segments on the left)
    M22 S = P;
    for (int d = 1; d < 32; d <<= 1) {
        const M22 o = m22_shfl(S, d, true);
        if (lane >= d) S = m22_mul(S, o);
    }
    const M22 Sprev = m22_shfl(S, 1, true);          // S_{k-1}
    float f0, f1;
    {
        const float w = chain[0];
        const float a0 = 1.f - w, a1 = w, sum = a0 + a1;
        f0 = a0 / sum;
        f1 = a1 / sum;
    }
    if (lane > 0) {                                   // f_{i0 - 1} = S_{k-1} f_0
        const float a0 = Sprev.a * f0 + Sprev.b * f1, a1 = Sprev.c * f0 + Sprev.d * f1, sum = a0 + a1;
        f0 = a0 / sum;
        f1 = a1 / sum;
    }
    if (has) {
        int i = i0;
        if (i == 0) {
            fw[0] = make_float2(f0, f1);
            i = 1;
        }
        for (; i < i1; ++i) {
            const float w = e[i - i0];
            const float p0 = g * f0 + h * f1, p1 = h * f0 + g * f1;
            const float a0 = (1.f - w) * p0, a1 = w * p1, sum = a0 + a1;
            f0 = a0 / sum;
            f1 = a1 / sum;
            fw[i - i0] = make_float2(f0, f1);
        }
    }

    // ---- backward: segment products of A diag(e_{i+1}) for i in [i0, min(i1, len - 1))
    const int j1 = min(i1, len - 1);
    M22 R{1.f, 0.f, 0.f, 1.f};
    for (int i = j1 - 1; i >= i0; --i) {
        const float w = i + 1 < i1 ? e[i + 1 - i0] : e[LP];
        const M22 Ni{g * (1.f - w), h * w, h * (1.f - w), g * w};
        R = m22_mul(Ni, R);                           // N_i ... N_{j1 - 1}
    }
    // the emission just past this segment, read before any lane writes q
    const float w_after = i1 < len ? e[LP] : 0.f;
    // suffix scan: U_k = R_k R_{k+1} ... R_31
    M22 U = R;
    for (int d = 1; d < 32; d <<= 1) {
        const M22 o = m22_shfl(U, d, false);
        if (lane + d < 32) U = m22_mul(U, o);
    }
    const M22 Unext = m22_shfl(U, 1, false);          // U_{k+1}
    float b0 = 1.f, b1 = 1.f;                          // b_{len - 1}
    if (lane < 31 && i1 < len) {                       // b_{i1} = U_{k+1} 1
        const float n0 = Unext.a + Unext.b, n1 = Unext.c + Unext.d, sum = n0 + n1;
        b0 = n0 / sum;
        b1 = n1 / sum;
    }
    __syncwarp();                                      // every lane has read its emissions
    if (has) {
        float w_next = w_after;
        int i = i1 - 1;
        if (i1 == len) {                               // the chain's last element: b = 1
            w_next = e[i - i0];
            const float2 f = fw[i - i0];
            const float q0 = f.x * b0, q1 = f.y * b1;
            e[i - i0] = q1 / (q0 + q1);
            --i;
        }
        for (; i >= i0; --i) {
            const float c0 = (1.f - w_next) * b0, c1 = w_next * b1;
            const float n0 = g * c0 + h * c1, n1 = h * c0 + g * c1, sum = n0 + n1;
            b0 = n0 / sum;
            b1 = n1 / sum;
            w_next = e[i - i0];
            const float2 f = fw[i - i0];
            const float q0 = f.x * b0, q1 = f.y * b1;
            e[i - i0] = q1 / (q0 + q1);
        }
    }
}

// grid (groups of chains, frame)
__global__ void __launch_bounds__(32 * kFbMaxWarps) k_forward_backward(DevParams p, DevState s)
{
    extern __shared__ float fb_smem[];
    const int dir = (*s.iter) & 3;
    const bool rows = (dir == 0 || dir == 2);
    const int n_chains = rows ? p.H : p.W;
    const int len = rows ? p.W : p.H;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int per = fb_chains(len, max(p.W, p.H), blockDim.x >> 5), c0 = blockIdx.x * per, here = min(per, n_chains - c0);
    if (here <= 0) return;
    const int L = fb_segment(len), LP = L | 1, row = fb_row(len);
    float* q = s.qs + (size_t)blockIdx.y * p.N + (rows ? (size_t)c0 * p.W : (size_t)c0);
    // element i of chain k: es(k)[i + (i / L) (LP - L)]
    auto for_all = [&](auto&& f) {
        if (rows) {
            if (warp < here)
                for (int i = lane; i < len; i += 32) f(q + (size_t)warp * p.W + i, fb_smem + 3 * row * warp + i + i / L * (LP - L));
        } else {
            for (int n = threadIdx.x; n < len * per; n += blockDim.x) {
                const int i = n / per, k = n % per;
                if (k < here) f(q + (size_t)i * p.W + k, fb_smem + 3 * row * k + i + i / L * (LP - L));
            }
        }
    };
    for_all([](float* g, float* m) { *m = *g; });
    __syncthreads();
    if (warp < here) {
        float* es = fb_smem + 3 * row * warp;
        fb_chain(p, len, es + lane * LP, reinterpret_cast<float2*>(es + row) + lane * LP, es);
    }
    __syncthreads();
    for_all([](float* g, float* m) { *g = *m; });
}

void launch_forward_backward(const DevParams& p, const DevState& s, cudaStream_t st)
{
    const int most = p.H > p.W ? p.H : p.W;               // chains in one direction, their length in the other
    const int smem = kFbChains * 3 * fb_row(most) * (int)sizeof(float);
    // the longest chain's, whatever this window's: the attribute belongs to all windows and threads
    constexpr int kSmemMax = kFbChains * 3 * fb_row(kMaxImageSide) * (int)sizeof(float);
    cudaFuncSetAttribute(k_forward_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    const int warps = fb_warps(most, std::min(p.W, p.H));
    const int rows = fb_chains(p.W, most, warps), cols = fb_chains(p.H, most, warps);   // chains to a block, along rows and columns
    const int blocks = std::max((p.H + rows - 1) / rows, (p.W + cols - 1) / cols);
    k_forward_backward<<<dim3(blocks, p.T), 32 * warps, smem, st>>>(p, s);
}

}  // namespace vd
