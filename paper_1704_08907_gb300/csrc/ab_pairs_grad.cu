// Pair sums, adjoints: the Gaussian and Lennard-Jones gradients, with or without
// the values in the same walk (see ab_pairs.cuh).
#include "ab_pairs.cuh"

namespace ab {

namespace {

// Adjoints (GAUSS, LJ): direct visit.  (A batched variant that collected
// acceptances in a per-lane bit mask and evaluated the bodies when draining
// it measured 6-15% slower once the predicate was packed.)
// DS (GAUSS): the partials of ds are wanted.
// VALUE: the forward value of the same operator in the same walk (the
// upstream gradient is known when the forward runs); each forward term is
// the forward kernel's expression, accumulated in the same visit order, so
// both outputs equal the separate kernels' bit for bit.  With VALUE the
// partials carry the LJ energy (GAUSS: still ds).
template <int DIM, int MODE, int SL, int OP, bool VALUE, bool DS>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_bwd(PairParams P, PairOut o) {
    allow_dependents();
    wait_prerequisite();
    uint32_t sub;
    const uint32_t s = pair_particle<SL>(sub);
    const bool live = s < P.n;
    const float4 pi = live ? __ldg(P.spos + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    // the upstream gradient g rides in the pad component of the sorted
    // positions; GAUSS also needs w: in 2-D in the unused third component, in
    // 3-D a float per particle (sv as float[n])
    const float* __restrict__ wv = reinterpret_cast<const float*>(P.sv);
    const float wi = OP != AB_OP_GAUSS ? 0.0f : DIM == 2 ? pi.z : live ? __ldg(wv + s) : 0.0f;
    float gx = 0.0f, gy = 0.0f, gz = 0.0f, dw = 0.0f, ds = 0.0f, y = 0.0f;
    if (live) visit_pairs<DIM, MODE, 4, SL>(P, s, sub, pi,
        [&](uint32_t j, const float4& pj, float dx, float dy, float dz, float d2) {
            if (OP == AB_OP_GAUSS) {
                const float wj = DIM == 2 ? pj.z : __ldg(wv + j);
                const float k = ex2_approx(-P.s_log2e * d2);
                if (VALUE) y = fmaf(wj, k, y);
                const float coef = fmaf(pi.w, wj, pj.w * wi) * k;
                gx = fmaf(coef, dx, gx);
                gy = fmaf(coef, dy, gy);
                if (DIM == 3) gz = fmaf(coef, dz, gz);
                dw = fmaf(pj.w, k, dw);
                if (DS) ds = fmaf(wj * k, d2, ds);
            } else {  // LJ: 1/2 (g_i + g_j) eps (12 sr12 - 6 sr6) / d2
                const float inv = rcp_approx(d2);
                const float sr2 = P.sig2 * inv;
                const float sr6 = sr2 * sr2 * sr2;
                if (VALUE) y = fmaf(sr6, sr6 - 1.0f, y);
                const float coef = (pi.w + pj.w) * (sr6 * fmaf(6.0f, sr6, -3.0f)) * inv;
                gx = fmaf(coef, dx, gx);
                gy = fmaf(coef, dy, gy);
                if (DIM == 3) gz = fmaf(coef, dz, gz);
            }
        });
    gx = lane_sum<SL>(gx);
    gy = lane_sum<SL>(gy);
    if (DIM == 3) gz = lane_sum<SL>(gz);
    if (OP == AB_OP_GAUSS) {
        dw = lane_sum<SL>(dw);
        if (DS) ds = lane_sum<SL>(ds);
    }
    if (VALUE) y = lane_sum<SL>(y);
    if (VALUE && OP == AB_OP_LJ) y *= 0.5f * P.eps;
    const bool lead = live && sub == 0;
    if (lead) {
        const uint32_t p = __ldg(P.perm + s);
        if (VALUE && o.out) o.out[p] = y;
        if (OP == AB_OP_GAUSS) {
            const float two_s = 2.0f * P.s;
            if (o.grad_pos)
                o.grad_pos[p] = make_float4(two_s * gx, two_s * gy,
                                            DIM == 3 ? two_s * gz : 0.0f, 0.0f);
            if (o.grad_w) o.grad_w[p] = dw;
        } else if (o.grad_pos) {
            o.grad_pos[p] = make_float4(P.eps * gx, P.eps * gy, DIM == 3 ? P.eps * gz : 0.0f, 0.0f);
        }
    }
    if (OP == AB_OP_GAUSS && DS)
        block_partial<kPairThreads>(lead ? -(double)pi.w * (double)ds : 0.0, o.partial);
    if (VALUE && OP == AB_OP_LJ && o.partial)
        block_partial<kPairThreads>(lead ? (double)y : 0.0, o.partial);
}

// LJ energy and its gradient in one walk, for a loss equal to the total
// energy (every per-particle energy has upstream gradient 1): the forward's
// E_i = 1/2 eps sum_j ((sig/d)^12 - (sig/d)^6) and the adjoint's
// dE/dx_i = eps sum_j (g_i + g_j) C_ij dx_ij with g = 1, sharing the
// predicate and the powers of sig/d.  Bit for bit the results of k_pair_fwd_q
// (LJ) and of k_pair_bwd (LJ) with g = 1: the same visit order, the same
// expressions, and (g_i + g_j) = 2 exactly.
template <int DIM, int MODE, int SL>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_lj_eg(PairParams P, PairOut o) {
    allow_dependents();
    wait_prerequisite();
    uint32_t sub;
    const uint32_t s = pair_particle<SL>(sub);
    const bool live = s < P.n;
    const float4 pi = live ? __ldg(P.spos + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    float e = 0.0f, gx = 0.0f, gy = 0.0f, gz = 0.0f;
    if (live) visit_pairs<DIM, MODE, 2, SL>(P, s, sub, pi,
        [&](uint32_t, const float4&, float dx, float dy, float dz, float d2) {
            const float inv = rcp_approx(d2);
            const float sr2 = P.sig2 * inv;
            const float sr6 = sr2 * sr2 * sr2;
            e = fmaf(sr6, sr6 - 1.0f, e);
            // (g_i + g_j) (sr6 (6 sr6 - 3)) / d2 with g = 1: the factor 2 is
            // folded into the fma, exactly (scaling by 2 commutes with
            // rounding; 6 sr6 - 3 is 0 or far from the subnormal range)
            const float coef = (sr6 * fmaf(12.0f, sr6, -6.0f)) * inv;
            gx = fmaf(coef, dx, gx);
            gy = fmaf(coef, dy, gy);
            if (DIM == 3) gz = fmaf(coef, dz, gz);
        });
    e = lane_sum<SL>(e);
    gx = lane_sum<SL>(gx);
    gy = lane_sum<SL>(gy);
    if (DIM == 3) gz = lane_sum<SL>(gz);
    const bool lead = live && sub == 0;
    if (lead) {
        const uint32_t p = __ldg(P.perm + s);
        e *= 0.5f * P.eps;
        if (o.out) o.out[p] = e;
        if (o.grad_pos)
            o.grad_pos[p] = make_float4(P.eps * gx, P.eps * gy, DIM == 3 ? P.eps * gz : 0.0f, 0.0f);
        if (o.grad_packed) {   // DIM floats per particle
            float* q = o.grad_packed + (int64_t)p * DIM;
            q[0] = P.eps * gx;
            q[1] = P.eps * gy;
            if (DIM == 3) q[2] = P.eps * gz;
        }
    }
    if (o.partial) block_partial<kPairThreads>(lead ? (double)e : 0.0, o.partial);
}

}  // namespace

cudaError_t launch_pair_bwd(const CellList& cl, ab_op op, const ab_op_params& prm,
                            const float2* sv, PairOut& o, cudaStream_t st, bool value) {
    if (cl.n <= 0) return cudaSuccess;
    const PairParams P = make_params(cl, op, prm, sv);
    const bool ds = o.partial != nullptr;
    switch (op) {
        case AB_OP_GAUSS:
            if (value)
                return ds ? AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_GAUSS, true, true>)
                          : AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_GAUSS, true, false>);
            return ds ? AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_GAUSS, false, true>)
                      : AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_GAUSS, false, false>);
        case AB_OP_LJ:
            return value ? AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_LJ, true, false>)
                         : AB_PAIR_LAUNCH(k_pair_bwd<DIM, MODE, SL, AB_OP_LJ, false, false>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_pair_energy_grad(const CellList& cl, ab_op op, const ab_op_params& prm,
                                   PairOut& o, cudaStream_t st) {
    if (cl.n <= 0) return cudaSuccess;
    if (op != AB_OP_LJ) return cudaErrorNotSupported;
    const PairParams P = make_params(cl, op, prm, nullptr);
    return AB_PAIR_LAUNCH(k_pair_lj_eg<DIM, MODE, SL>);
}

}  // namespace ab
