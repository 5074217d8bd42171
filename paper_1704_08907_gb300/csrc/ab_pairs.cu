// Pair sums, values: every operator's forward, the neighbour count and the
// neighbour list (see ab_pairs.cuh).
#include "ab_pairs.cuh"

namespace ab {

namespace {

// Forward for the cheap operators (COUNT, GAUSS, SPH density): direct visit.
// The weight w_j (GAUSS) or mass m_j (SPH) comes in the pad component of the
// sorted position, loaded with the candidate.  RARE (SPH): few candidates are
// neighbours (see visit_pairs).
template <int DIM, int MODE, int SL, int OP, bool RARE = false>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_fwd(PairParams P, PairOut o) {
    wait_prerequisite();
    uint32_t sub;
    const uint32_t s = pair_particle<SL>(sub);
    const bool live = s < P.n;
    if (SL == 0 && !live) return;
    const float4 pi = live ? __ldg(P.spos + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    float a0 = 0.0f;
    if (live) visit_pairs<DIM, MODE, 2, SL>(P, s, sub, pi,
        [&](uint32_t, const float4& pj, float, float, float, float d2) {
            if (OP == AB_OP_COUNT) {
                a0 += 1.0f;
            } else if (OP == AB_OP_GAUSS) {
                a0 = fmaf(pj.w, ex2_approx(-P.s_log2e * d2), a0);
            } else {   // SPH_DENSITY: m_j W(d) / a
                // (1 - q)^4 (1 + 4 q), q = d / r, in t = 1 - q
                const float t = fmaf(-P.inv_r, pair_distance<RARE>(d2), 1.0f), t2 = t * t;
                a0 = fmaf(pj.w, t2 * t2 * fmaf(-4.0f, t, 5.0f), a0);
            }
        });
    a0 = lane_sum<SL>(a0);
    if (SL > 0 && (!live || sub != 0)) return;
    if (OP == AB_OP_SPH_DENSITY) a0 = (a0 + pi.w) * P.wend_a;   // with the particle itself
    o.out[__ldg(P.perm + s)] = a0;
}

// Forward for LJ / EXPF / SOFT / SPH force: direct visit.  RARE (SPH force): few
// candidates are neighbours (see visit_pairs).
template <int DIM, int MODE, int SL, int OP, bool RARE = false>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_fwd_q(PairParams P, PairOut o) {
    allow_dependents();
    wait_prerequisite();
    uint32_t sub;
    const uint32_t s = pair_particle<SL>(sub);
    const bool live = s < P.n;
    const float4 pi = live ? __ldg(P.spos + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
    const float ai = OP != AB_OP_SPH_FORCE ? 0.0f : DIM == 2 ? pi.w : live ? __ldg(&P.sv[s].y) : 0.0f;
    if (live) visit_pairs<DIM, MODE, (OP == AB_OP_EXPF || OP == AB_OP_SOFT || RARE) ? 4 : 2, SL>(P, s, sub, pi,
        [&](uint32_t j, const float4& pj, float dx, float dy, float dz, float d2) {
            // EXPF and the SPH force leave out their common factor P.fscale
            // (one multiplication a particle instead of one a pair; SOFT
            // keeps its rounding, see pair_lanes_log2), and in 2-D
            // the third component, which the compiler cannot drop
            // (0 mag may be NaN)
            float mag;
            if (OP == AB_OP_LJ) {
                const float sr2 = P.sig2 * rcp_approx(d2);
                const float sr6 = sr2 * sr2 * sr2;
                a0 = fmaf(sr6, sr6 - 1.0f, a0);
                return;
            } else if (OP == AB_OP_SPH_FORCE) {
                // m_j (A_i + A_j) c^3 (1 - d/r)^3 dx
                const float2 vj = DIM == 2 ? make_float2(pj.z, pj.w) : __ldg(P.sv + j);
                const float t = fmaf(-P.grad_c_inv_r, pair_distance<RARE>(d2), P.grad_c);
                mag = vj.x * (ai + vj.y) * (t * t * t);
            } else {
                // coincident points contribute 0: a finite mag times 0
                const float inv_d = rsqrt_approx(fmaxf(d2, 1.17549435e-38f));
                const float d = d2 * inv_d;
                // SOFT: (r - d) / d with r - d = (r^2 - d^2) / (r + d): the fma
                // rounds r^2 - d^2 once, so the term keeps its relative
                // accuracy up to the cut-off, where r - d cancels, and d
                // enters only through 1/d and r + d (approximate
                // reciprocals, a few ulp)
                if (OP == AB_OP_EXPF) mag = ex2_approx(-kLog2e * d) * inv_d;
                else mag = (-P.k * fmaf(P.r, P.r, -d2)) * (inv_d * rcp_approx(P.r + d));
            }
            a0 = fmaf(mag, dx, a0);
            a1 = fmaf(mag, dy, a1);
            if (DIM == 3) a2 = fmaf(mag, dz, a2);
        });
    a0 = lane_sum<SL>(a0);
    if (OP != AB_OP_LJ) {
        a1 = lane_sum<SL>(a1);
        if (DIM == 3) a2 = lane_sum<SL>(a2);
    }
    const bool lead = live && sub == 0;
    if (lead) {
        const uint32_t p = __ldg(P.perm + s);
        if (OP == AB_OP_LJ) {
            a0 *= 0.5f * P.eps;
            o.out[p] = a0;
        } else {
            // a sum without terms (or of coincident points alone) stays 0 also
            // where the factor is infinite
            auto scaled = [&](float a) { return a == 0.0f ? 0.0f : P.fscale * a; };
            o.out4[p] = make_float4(scaled(a0), scaled(a1), DIM == 3 ? scaled(a2) : 0.0f, 0.0f);
        }
    }
    if (OP == AB_OP_LJ && o.partial) block_partial<kPairThreads>(lead ? (double)a0 : 0.0, o.partial);
}

template <int DIM, int MODE, int SL>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_count(PairParams P, uint32_t* __restrict__ counts) {
    wait_prerequisite();
    uint32_t sub;
    const uint32_t s = pair_particle<SL>(sub);
    const bool live = s < P.n;
    if (SL == 0 && !live) return;
    const float4 pi = live ? __ldg(P.spos + s) : make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t c = 0;
    if (live) visit_pairs<DIM, MODE, 2, SL>(P, s, sub, pi,
        [&](uint32_t, const float4&, float, float, float, float) { ++c; });
    c = lane_sum<SL>(c);
    if (SL > 0 && (!live || sub != 0)) return;
    counts[__ldg(P.perm + s)] = c;
}

template <int DIM, int MODE>
__global__ void __launch_bounds__(kPairThreads, 8)
k_pair_emit(PairParams P, const int64_t* __restrict__ offsets, int32_t* __restrict__ idx) {
    wait_prerequisite();
    const uint32_t s = blockIdx.x * kPairThreads + threadIdx.x;
    if (s >= P.n) return;
    const float4 pi = __ldg(P.spos + s);
    int64_t at = offsets[__ldg(P.perm + s)];
    visit_pairs<DIM, MODE, 2, 0>(P, s, 0u, pi,
        [&](uint32_t j, const float4&, float, float, float, float) {
            idx[at++] = (int32_t)__ldg(P.perm + j);
        });
}

}  // namespace

int pair_grid(const CellList& cl) { return pair_blocks(cl, pair_lanes_log2(cl, AB_OP_LJ)); }

size_t pair_partial_capacity(int64_t n) {
    const int64_t split = n < kMaxSplitN ? n : kMaxSplitN;
    const int64_t threads = n > split << kMaxLanesLog2 ? n : split << kMaxLanesLog2;
    return (size_t)((threads + kPairThreads - 1) / kPairThreads);
}

cudaError_t launch_pair_fwd(const CellList& cl, ab_op op, const ab_op_params& prm,
                            const float2* sv, PairOut& o, cudaStream_t st) {
    if (cl.n <= 0) return cudaSuccess;
    const PairParams P = make_params(cl, op, prm, sv);
    switch (op) {
        case AB_OP_COUNT: return AB_PAIR_LAUNCH(k_pair_fwd<DIM, MODE, SL, AB_OP_COUNT>);
        case AB_OP_GAUSS: return AB_PAIR_LAUNCH(k_pair_fwd<DIM, MODE, SL, AB_OP_GAUSS>);
        case AB_OP_LJ: return AB_PAIR_LAUNCH(k_pair_fwd_q<DIM, MODE, SL, AB_OP_LJ>);
        case AB_OP_EXPF: return AB_PAIR_LAUNCH(k_pair_fwd_q<DIM, MODE, SL, AB_OP_EXPF>);
        case AB_OP_SOFT: return AB_PAIR_LAUNCH(k_pair_fwd_q<DIM, MODE, SL, AB_OP_SOFT>);
        case AB_OP_SPH_DENSITY:
            if (pairs_are_rare(cl)) return AB_PAIR_LAUNCH(k_pair_fwd<DIM, MODE, SL, AB_OP_SPH_DENSITY, DIM == 3 && SL == 0>);
            return AB_PAIR_LAUNCH(k_pair_fwd<DIM, MODE, SL, AB_OP_SPH_DENSITY>);
        case AB_OP_SPH_FORCE:
            if (pairs_are_rare(cl)) return AB_PAIR_LAUNCH(k_pair_fwd_q<DIM, MODE, SL, AB_OP_SPH_FORCE, DIM == 3 && SL == 0>);
            return AB_PAIR_LAUNCH(k_pair_fwd_q<DIM, MODE, SL, AB_OP_SPH_FORCE>);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_pair_count(const CellList& cl, uint32_t* counts, cudaStream_t st) {
    if (cl.n <= 0) return cudaSuccess;
    const ab_op op = AB_OP_COUNT;
    const PairParams P = make_params(cl, op, ab_op_params{}, nullptr);
    uint32_t* const o = counts;
    return AB_PAIR_LAUNCH(k_pair_count<DIM, MODE, SL>);
}

// One lane a particle: the indices come out in traversal order.
cudaError_t launch_pair_emit(const CellList& cl, const int64_t* offsets, int32_t* idx,
                             cudaStream_t st) {
    if (cl.n <= 0) return cudaSuccess;
    const PairParams P = make_params(cl, AB_OP_COUNT, ab_op_params{}, nullptr);
    const int grid = (int)((cl.n + kPairThreads - 1) / kPairThreads);
    auto emit = [&](auto dim) {
        constexpr int DIM = decltype(dim)::value;
        auto* fn = cl.g.general ? k_pair_emit<DIM, kModeGeneral>
                   : cl.g.compact ? k_pair_emit<DIM, kModeCompact>
                                  : k_pair_emit<DIM, kModeFast>;
        return pdl_launch(fn, grid, kPairThreads, st, P, offsets, idx);
    };
    return cl.g.dim == 3 ? emit(std::integral_constant<int, 3>{}) : emit(std::integral_constant<int, 2>{});
}

}  // namespace ab
