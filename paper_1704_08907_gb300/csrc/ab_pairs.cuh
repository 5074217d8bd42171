// Shared by the pair kernels of ab_pairs.cu (values) and ab_pairs_grad.cu
// (adjoints): the stencil walk, the exact neighbour predicate and the dispatch.
//
// Fixed-radius pair sums over the cell list (paper Sec. 2.2.2 box search:
// a particle's cell and its adjacent cells; Sec. 3, Eq. 1 and the velocity-
// update listing: the radius-filtered sum over the shortest separation).
//
// One thread per sorted particle i.  Sorted order puts the particles of one
// cell in consecutive threads, so a warp walks the same few neighbour cells
// and the float4 neighbour loads hit L1.  Along x the three stencil cells of
// a row are contiguous in sorted order, so a 3-D stencil is 9 row segments
// (plus one extra segment where a row wraps through a periodic face).
//
// Exact neighbour predicate.  The canonical rule (also the oracle's) is
//   dx = fl(x_j - x_i); periodic axis: dx > L/2 -> fl(dx - L),
//                                      dx < -L/2 -> fl(dx + L);
//   d2 = fl(fl(fl(dx0*dx0) + fl(dx1*dx1)) + fl(dx2*dx2)); pair iff d2 < r2.
// The __fsub_rn/__fmul_rn/__fadd_rn intrinsics are never contracted into FMA.
// Fast path: when every periodic axis has >= 5 cells the wrap decision is
// fixed per stencil cell -- a neighbour cell reached through the face is at
// least 3 cells (> L/2) away the other way, and one reached directly is at
// most 2 cells (< L/2) away -- so dx = fl(fl(x_j - x_i) + shift) with a
// per-segment shift in {-L, 0, +L} is bit-identical to the canonical rule
// (adding 0 is exact).  Otherwise the kernel applies the canonical rule per
// candidate (GENERAL).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "ab_internal.cuh"

namespace ab {

namespace {

constexpr int kPairThreads = 128;
constexpr float kLog2e = 1.4426950408889634f;

struct PairParams {
    const float4* __restrict__ spos;
    const uint32_t* __restrict__ cell_start;   // dense: per cell; compact: per occupied cell
    const uint4* __restrict__ occ;             // compact: occupancy words (see cell_bound)
    const uint32_t* __restrict__ perm;
    const float2* __restrict__ sv;
    int64_t n;
    Geom g;
    float s, s_log2e, eps, sig2, k, r;
    float fscale;         // factor of a vector sum: -c (EXPF), a power of two (SOFT), within [1, 8] (SPH force)
    float zero;   // 0.0f, passed at run time (see sq2)
    float wend_a;         // Wendland C2 normalisation a (SPH)
    float inv_r;          // 1 / r
    float grad_c, grad_c_inv_r;   // SPH force: a power of two c, c^3 about 20 a / r^2, and c / r
};


__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Distance of a pair at d^2, 0 for coincident points: with a floor that keeps
// the reciprocal root finite, one operation where a test and a select take two,
// or (BRANCH) with the test, beside which the compiler leaves the body behind a
// branch instead of issuing it under a predicate on every candidate.  The same
// bits.
template <bool BRANCH>
__device__ __forceinline__ float pair_distance(float d2) {
    if (BRANCH) return d2 > 0.0f ? d2 * rsqrt_approx(d2) : 0.0f;
    return d2 * rsqrt_approx(fmaxf(d2, 1.17549435e-38f));
}

// Canonical FP32 minimum image along one periodic axis.
__device__ __forceinline__ float min_image(float d, float L, float halfL) {
    if (d > halfL) return __fsub_rn(d, L);
    if (d < -halfL) return __fadd_rn(d, L);
    return d;
}

// One neighbour coordinate along axis k for offset o (|o| <= reach): returns
// false if the offset leaves a non-periodic box or repeats a cell already
// visited (periodic axes with fewer than 3 cells, general path only);
// *shift receives the fast-path shift (-L when reaching through the lower
// face, +L through the upper face; meaningful when every periodic axis has
// at least 2 reach + 3 cells).
__device__ __forceinline__ bool stencil_coord(const Geom& g, int k, int c, int o, int& t,
                                              float& shift) {
    const int n = g.n[k];
    t = c + o;
    shift = 0.0f;
    if (!g.periodic[k]) return t >= 0 && t < n;
    if (n == 1) return o == 0;
    if (n == 2) {                 // cells {0, 1}: offsets 0 and +1 cover both
        if (o == -1) return false;
        t = (c + o) & 1;
        return true;
    }
    if (t < 0) { t += n; shift = -g.L[k]; }
    else if (t >= n) { t -= n; shift = g.L[k]; }
    return true;
}

// Value separation along one axis, accurate to one rounding: the canonical
// minimum image of x_j - x_i, where a wrapped difference is corrected by the
// rounding error of fl(x_j - x_i) (Knuth's TwoSum).  fl(x_j - x_i) has
// magnitude above L/2 when it wraps, so fl(. -+ L) is exact (Sterbenz) and
// only the final addition of the error term rounds.  Without the correction
// a pair straddling a periodic face would carry an absolute error of
// ulp(L)/2 in a separation of size ~r.  The neighbour predicate never uses
// this value; it uses the canonical FP32 rule only.
__device__ __forceinline__ float two_sum_err(float a, float b, float s) {
    const float bp = __fsub_rn(s, a);
    const float ap = __fsub_rn(s, bp);
    return __fadd_rn(__fsub_rn(a, ap), __fsub_rn(b, bp));
}

__device__ __forceinline__ float value_sep(float xi, float xj, bool periodic, float L,
                                           float halfL) {
    const float s = __fsub_rn(xj, xi);
    if (periodic && (s > halfL || s < -halfL)) {
        const float e = two_sum_err(xj, -xi, s);
        const float w = (s > halfL) ? __fsub_rn(s, L) : __fadd_rn(s, L);
        return __fadd_rn(w, e);
    }
    return s;
}

// Kernel modes: the fast path over a dense cell table, the general path
// (canonical wrap per candidate, dense table), and the fast path over the
// compacted table of occupied cells.
constexpr int kModeFast = 0, kModeGeneral = 1, kModeCompact = 2;

// First sorted slot of cell c (c = n_cells gives n).  Dense table: one load.
// Compacted table: occ[c / 64] packs the occupancy bits of cells 64w ..
// 64w + 63 (x, y) and the number of occupied cells before them (z); the
// occupied cells before c index the compact offsets (an empty cell starts
// where the next occupied one does).
template <int MODE>
__device__ __forceinline__ uint32_t cell_bound(const PairParams& P, int64_t c) {
    if (MODE != kModeCompact) return __ldg(P.cell_start + c);
    const uint4 q = __ldg(P.occ + (c >> 6));
    const uint64_t bits = ((uint64_t)q.y << 32) | q.x;
    const uint32_t rank = q.z + (uint32_t)__popcll(bits & ((1ull << (c & 63)) - 1ull));
    return __ldg(P.cell_start + rank);
}

// Walk the stencil of the particle at pi: seg(a, b, sx, sy, sz) is called for
// each contiguous range [a, b) of sorted particles with its fast-path shift.
// Rows along x are contiguous in sorted order; a row that wraps through the
// periodic x face splits into two segments.
template <int DIM, int MODE, class S>
__device__ __forceinline__ void for_each_segment(const PairParams& P, const float4& pi,
                                                 S&& seg) {
    constexpr bool GENERAL = MODE == kModeGeneral;
    const Geom& g = P.g;
    const int cx = cell_coord(pi.x, g.lo[0], g.inv_w[0], g.n[0]);
    const int cy = cell_coord(pi.y, g.lo[1], g.inv_w[1], g.n[1]);
    const int cz = DIM == 3 ? cell_coord(pi.z, g.lo[2], g.inv_w[2], g.n[2]) : 0;
    const int nx = g.n[0];
    // x segments: [xa0, xb0] with shift xs0, optional [xa1, xb1] with xs1;
    // the stencil reaches kx cells each way along x (kx = 1 on the general
    // path)
    const int kx = GENERAL ? 1 : g.kx;
    int xa0, xb0, xa1 = 0, xb1 = -1;
    float xs0 = 0.0f, xs1 = 0.0f;
    if (!g.periodic[0]) {
        xa0 = cx > kx - 1 ? cx - kx : 0;
        xb0 = cx < nx - kx ? cx + kx : nx - 1;
    } else if (nx <= 3) {
        xa0 = 0;
        xb0 = nx - 1;
    } else if (cx - kx < 0) {
        xa0 = 0; xb0 = cx + kx; xa1 = nx - (kx - cx); xb1 = nx - 1; xs1 = GENERAL ? 0.0f : -g.L[0];
    } else if (cx + kx >= nx) {
        xa0 = cx - kx; xb0 = nx - 1; xa1 = 0; xb1 = cx + kx - nx; xs1 = GENERAL ? 0.0f : g.L[0];
    } else {
        xa0 = cx - kx; xb0 = cx + kx;
    }
    const int ky = GENERAL ? 1 : g.ky, kz = GENERAL ? 1 : g.kz;
#pragma unroll 1
    for (int oz = (DIM == 3 ? -kz : 0); oz <= (DIM == 3 ? kz : 0); ++oz) {
        int z = 0;
        float sz = 0.0f;
        if (DIM == 3 && !stencil_coord(g, 2, cz, oz, z, sz)) continue;
#pragma unroll 1
        for (int oy = -ky; oy <= ky; ++oy) {
            int y;
            float sy;
            if (!stencil_coord(g, 1, cy, oy, y, sy)) continue;
            if (GENERAL) sy = sz = 0.0f;
            const int64_t row = ((int64_t)z * g.n[1] + y) * nx;
            seg(cell_bound<MODE>(P, row + xa0), cell_bound<MODE>(P, row + xb0 + 1), xs0, sy, sz);
            if (xb1 >= xa1)
                seg(cell_bound<MODE>(P, row + xa1), cell_bound<MODE>(P, row + xb1 + 1), xs1, sy, sz);
        }
    }
}

// Packed FP32 pairs (sm_100+ f32x2 arithmetic; each half rounds exactly like
// the scalar FP32 instruction).  The x and y components of one float4 sit in
// an aligned register pair, so the predicate forms (dx, dy) and their squares
// with one instruction each.  Squares are fma(d, d, z) with z a zero known
// only at run time: rounded once, exactly like fl(d * d), and never
// contracted further with the following addition.
__device__ __forceinline__ uint64_t f2pack(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2unpack(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t sq2(uint64_t a, uint64_t z) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(d) : "l"(a), "l"(z));
    return d;
}

// Predicate separation (canonical FP32 rule) for candidate pj.
template <int DIM, bool GENERAL, bool SHIFTED>
__device__ __forceinline__ float pred_d2(const Geom& g, const float4& pi, const float4& pj,
                                         float sx, float sy, float sz, float& dx, float& dy,
                                         float& dz, float zero) {
    if (GENERAL) {
        dx = __fsub_rn(pj.x, pi.x);
        dy = __fsub_rn(pj.y, pi.y);
        dz = DIM == 3 ? __fsub_rn(pj.z, pi.z) : 0.0f;
        if (g.periodic[0]) dx = min_image(dx, g.L[0], g.halfL[0]);
        if (g.periodic[1]) dy = min_image(dy, g.L[1], g.halfL[1]);
        if (DIM == 3 && g.periodic[2]) dz = min_image(dz, g.L[2], g.halfL[2]);
        float d2 = __fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy));
        if (DIM == 3) d2 = __fadd_rn(d2, __fmul_rn(dz, dz));
        return d2;
    }
    uint64_t dxy = sub2(f2pack(pj.x, pj.y), f2pack(pi.x, pi.y));
    dz = DIM == 3 ? __fsub_rn(pj.z, pi.z) : 0.0f;
    if (SHIFTED) {
        dxy = add2(dxy, f2pack(sx, sy));
        if (DIM == 3) dz = __fadd_rn(dz, sz);
    }
    float qx, qy;
    f2unpack(sq2(dxy, f2pack(zero, zero)), qx, qy);
    f2unpack(dxy, dx, dy);
    float d2 = __fadd_rn(qx, qy);
    if (DIM == 3) d2 = __fadd_rn(d2, __fmul_rn(dz, dz));
    return d2;
}

// The kernels are bound by issue slots (29 instructions a candidate step in
// 3-D, the body entered on most of them by some lane), so a body's instruction
// count is its time.  What the bodies leave out, us before and after (SOFT /
// SPH density / SPH force / Gaussian adjoint): a common factor per pair, the
// third component in 2-D, tests for coincident points where a floor under the
// reciprocal root does, the clamp of 1 - d/r, ds where nobody asks for it, and
// in 2-D the second value's own load (it rides in the z component):
//   4M points in 2-D, 53 neighbours  406 / 493 / 558 / 550 -> 390 / 438 / 460 / 436
//   1M points in 3-D, 57 neighbours  344 / 358 / 422 / 391 -> 337 / 338 / 391 / 372
//   16.7M clustered points           5,129 / 5,375 / 6,554 / 5,871 -> 5,010 / 5,042 / 5,968 / 5,626
// (SOFT in 2-D with one special-function operation instead of two and three
// more FP32 ones: 417.  With its factor k taken out of the sum too: 381, 331
// and 4,886, not kept because it changes the last bits, see pair_lanes_log2.)
//
// Where few candidates are neighbours (cells wider than the cut-off, as when the
// table of a sparse or clustered input reaches its size limit: 2.6% of a stencil
// twice as wide, 21% else) the SPH bodies are better left behind a branch (see
// pair_distance), and the SPH force then unrolled by 4.  us, floor / branch (SPH
// force: and 4), 3-D points:
//   stencil 162 r^3  1M in 250 blobs  density 705 / 664   force 832 / 648
//                    250,000 in 62            257 / 246         297 / 249
//   stencil 20 r^3   16.7M in 1,024         5,090 / 5,046     6,050 / 6,500
//                    1M on a lattice          333 / 336         386 / 413
//   2-D              1M on a lattice          104 / 107         107 / 115
// so they branch where the stencil is larger than kRareStencil r^3 and a particle
// has one lane (with four, 50,000 points of which many crowd: force 65 / 85).
//
// Direct visit: f(j, pj, dx, dy, dz, d2) for every accepted pair, with value
// separations accurate to one rounding (see value_sep).  Used by every pair
// kernel.  UNROLL is the unroll factor of the candidate loop, measured per
// kernel: 2 where the body is short or rarely taken (forwards, COUNT, the
// fused LJ kernel), 4 for the adjoints and the EXPF / SOFT forces.
// SL > 0: the 2^SL lanes of a particle take its candidates in turn (lane `sub`
// of them the candidates a + sub, a + sub + 2^SL, ...).
template <int DIM, int MODE, int UNROLL, int SL, class F>
__device__ __forceinline__ void visit_pairs(const PairParams& P, uint32_t s, uint32_t sub,
                                            const float4& pi, F&& f) {
    constexpr uint32_t step = 1u << SL;
    constexpr bool GENERAL = MODE == kModeGeneral;
    const Geom& g = P.g;
    const float r2 = g.r2;
    for_each_segment<DIM, MODE>(P, pi, [&](uint32_t a0, uint32_t b0, float sx, float sy,
                                              float sz) {
      // the segment holding the particle itself is walked as [a0, s), (s, b0)
      uint32_t a = a0 + (SL ? sub : 0u), b = (a0 <= s && s < b0) ? s : b0;
      for (;;) {
        if (GENERAL || sx != 0.0f || sy != 0.0f || sz != 0.0f) {
#pragma unroll 1
            for (uint32_t j = a; j < b; j += step) {
                const float4 pj = __ldg(P.spos + j);
                float dx, dy, dz;
                const float d2 = pred_d2<DIM, GENERAL, true>(g, pi, pj, sx, sy, sz, dx, dy, dz, P.zero);
                if (d2 < r2) {
                    dx = value_sep(pi.x, pj.x, g.periodic[0], g.L[0], g.halfL[0]);
                    dy = value_sep(pi.y, pj.y, g.periodic[1], g.L[1], g.halfL[1]);
                    if (DIM == 3) dz = value_sep(pi.z, pj.z, g.periodic[2], g.L[2], g.halfL[2]);
                    f(j, pj, dx, dy, dz, fmaf(dz, dz, fmaf(dy, dy, dx * dx)));
                }
            }
        } else {
#pragma unroll (SL == 0 ? UNROLL : SL < 5 ? 2 : 4)
            for (uint32_t j = a; j < b; j += step) {
                const float4 pj = __ldg(P.spos + j);
                float dx, dy, dz;
                const float d2 = pred_d2<DIM, false, false>(g, pi, pj, 0.f, 0.f, 0.f, dx, dy, dz, P.zero);
                if (d2 < r2) f(j, pj, dx, dy, dz, d2);
            }
        }
        if (b >= b0) break;
        a = b + 1 + (SL ? sub : 0u);
        b = b0;
      }
    });
}

// Lets a programmatic dependent launch of the partials' reduction begin
// (its blocks then wait for this grid to finish): called at the start of
// every kernel that writes block partials.
__device__ __forceinline__ void allow_dependents() {
    asm volatile("griddepcontrol.launch_dependents;");
}

// Every pair kernel is a programmatic dependent launch of the kernel before
// it on the stream (normally the build): it may be scheduled while that
// kernel finishes, and waits here, before its first global read, until that
// grid has completed and its writes are visible.  Without a prerequisite
// grid the wait returns at once.
__device__ __forceinline__ void wait_prerequisite() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The particle of this thread, and its lane among the particle's.
template <int SL>
__device__ __forceinline__ uint32_t pair_particle(uint32_t& sub) {
    const uint32_t t = blockIdx.x * kPairThreads + threadIdx.x;
    sub = t & ((1u << SL) - 1u);
    return t >> SL;
}

// The sum over a particle's 2^SL lanes, in every one of them.  Called by whole
// warps.
template <int SL, class V>
__device__ __forceinline__ V lane_sum(V v) {
#pragma unroll
    for (int o = 1; o < (1 << SL); o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// FP64 block sum of one value per thread into partial[blockIdx.x].
template <int THREADS>
__device__ __forceinline__ void block_partial(double v, double* partial) {
    __shared__ double s_red[THREADS / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < THREADS / 32; ++w) t += s_red[w];
        partial[blockIdx.x] = t;
    }
}

// Volume of the stencil over r^3 in 3-D above which a pair is rare.
constexpr double kRareStencil = 70.0;
inline bool pairs_are_rare(const CellList& cl) {
    if (cl.g.dim != 3) return false;
    const int reach[3] = {cl.g.kx, cl.g.ky, cl.g.kz};
    double v = 1.0;
    for (int k = 0; k < 3; ++k) {
        const int cells = 2 * reach[k] + 1 < cl.g.n[k] ? 2 * reach[k] + 1 : cl.g.n[k];
        v *= (double)cells / cl.g.n[k] * cl.g.L[k] / cl.g.r;
    }
    return v > kRareStencil;
}

// Lanes that share a particle's walk (log2), the same for every table of a
// cell list and, but for SOFT and counts (exact in any order) in 2-D, for every
// operator, so that their results can be compared bit for bit.  SOFT drives
// time steppers in place: a last bit of a force moves a position by one, and a
// pair closer than some 30,000 of them then turns by more than a thousandth in
// the next step.  Points in the plane come that close by chance from about a
// hundred thousand of them, so there SOFT keeps one lane and the order of its
// sums.
// One lane a particle while the particles fill the SMs.  Fewer leave SMs
// idle, and one lane's walk, thousands of dependent loads on dense inputs, is
// all there is to wait for; more lanes then share it, but each row of a
// stencil costs a lane its set-up and a warp its longest lane, so short rows
// take fewer.  row: candidates expected in a stencil row.  Time over the best
// of the five, 1 / 2 / 4 / 8 / 32 lanes (geometric mean of EXPF, counts,
// Gaussian adjoint and fused LJ in 2-D and 3-D, uniform points):
//   row 1:    16,384 1.21/1.10/1.01/1.06/2.1    65,536 1.09/1.01/1.33/1.85/5.2
//   row 8:    16,384 1.83/1.33/1.07/1.00/1.9    65,536 1.26/1.02/1.10/1.32/3.8
//            120,000 1.06/1.03/1.16/1.56/5.0   196,608 1.03/1.08/1.35/1.93/6.7
//   row 25:   32,768 2.29/1.59/1.03/1.14/2.2    98,304 1.45/1.10/1.00/1.26/3.4
//            196,608 1.12/1.01/1.04/1.39/4.1   262,144 1.07/1.01/1.10/1.51/4.6
//   row 60:    8,192 3.84/2.45/1.47/1.05/1.04  196,608 1.18/1.08/1.01/1.16/2.8
//   row 130:  12,000 4.63/2.95/1.78/1.08/1.00   16,384 4.29/2.71/1.55/1.00/1.2
//             98,304 1.70/1.29/1.04/1.01/1.75  230,000 1.18/1.09/1.01/1.06/2.1
//   row 260:  16,384 5.74/3.76/2.11/1.21/1.00   65,536 2.18/1.58/1.24/1.00/1.2
//   row 500:  50,000 2.82/2.08/1.33/1.06/1.00  160,000 1.45/1.33/1.09/1.00/1.2
//   row 1000: 80,000 2.27/1.75/1.42/1.13/1.00
// Rows that are short on average may be long where points crowd, so up to
// 65,536 particles they keep more lanes than uniform points want: 50,000 points,
// a fiftieth of them at one place, density 48 us with four lanes and 173 with
// one, 65,536 uniform points with half a neighbour 27 and 19.
// Million-particle inputs lose 10-20% with two lanes already.
// No rule gives more than kMaxSplitN << kMaxLanesLog2 lanes in all, or a
// particle more than 2^kMaxLanesLog2 (pair_partial_capacity builds on it).
constexpr int64_t kMaxSplitN = 3 << 15;
constexpr int kMaxLanesLog2 = 5;
inline int pair_lanes_log2(const CellList& cl, ab_op op) {
    const int64_t n = cl.n;
    if (op == AB_OP_SOFT && cl.g.dim == 2 && n > 1 << 15) return 0;
    // counts have the shortest body: 250,000 points in 2-D with 600 neighbours 192
    // us with four lanes, 176 with one (3-D, 340: 299 and 373)
    if (op == AB_OP_COUNT && cl.g.dim == 2 && n > 3 << 16) return 0;
    const double row = (double)n / (double)cl.g.n_cells * (2 * cl.g.kx + 1);
    if (n > (1 << 18)) return 0;
    if (row >= 100.0) {
        if (n <= kMaxSplitN && (double)n <= 125.0 * row) return kMaxLanesLog2;
        return n <= 3 << 16 ? 3 : 2;
    }
    if (row >= 12.0) {
        if (n <= 1 << 13) return row >= 40.0 ? 5 : 3;
        if (n <= 1 << 15) return 3;
        return n <= 1 << 17 || row >= 40.0 ? 2 : 1;
    }
    return n <= 1 << 14 ? 3 : n <= 1 << 16 ? 2 : 0;
}

inline PairParams make_params(const CellList& cl, ab_op op, const ab_op_params& prm, const float2* sv) {
    PairParams P;
    P.spos = cl.spos;
    P.cell_start = cl.cell_start;
    P.occ = cl.occ;
    P.perm = cl.perm;
    P.sv = sv;
    P.n = cl.n;
    P.g = cl.g;
    P.s = prm.s;
    P.s_log2e = prm.s * kLog2e;
    P.eps = prm.eps;
    P.sig2 = prm.sigma * prm.sigma;
    P.k = prm.k;
    P.r = cl.g.r;
    P.zero = 0.0f;
    const double r = (double)cl.g.r, pi = 3.14159265358979323846;
    const double a = cl.g.dim == 3 ? 21.0 / (2.0 * pi * r * r * r) : 7.0 / (pi * r * r);
    P.wend_a = (float)a;
    P.inv_r = (float)(1.0 / r);
    // W'(d)/d = -20 a / r^2 (1 - d/r)^3: its power of two lies within the cube, (c
    // - c d/r)^3, which costs a pair nothing and keeps the terms in range; the rest
    // is the sum's
    const double f = 20.0 * a / (r * r);
    int e = (int)floor(log2(f) / 3.0);
    e = e < -40 ? -40 : e > 40 ? 40 : e;
    P.grad_c = ldexpf(1.0f, e);
    P.grad_c_inv_r = P.inv_r * P.grad_c;
    P.fscale = op == AB_OP_EXPF ? -prm.c : op == AB_OP_SOFT ? 1.0f : (float)(-ldexp(f, -3 * e));
    if (op == AB_OP_SOFT) {
        // A coincident pair meets k r / FLT_MIN^(1/2) before its separation of
        // 0.  Where that could overflow (k r > 3.7e19), a power of two is taken
        // out of k and put back at the end, which changes no rounding.
        const double top = fabs((double)prm.k) * (r > 1.0 ? r * r : r);
        if (!isfinite(prm.k)) {
            P.k = 1.0f;
            P.fscale = prm.k;
        } else if (top > 0x1p60) {
            int up = ilogb(top) - 59;
            if (up > 126) up = 126;
            P.k = ldexpf(prm.k, -up);
            P.fscale = ldexpf(1.0f, up);
        }
    }
    return P;
}

// Blocks of a pair kernel.
inline int pair_blocks(const CellList& cl, int lanes_log2) {
    return (int)(((cl.n << lanes_log2) + kPairThreads - 1) / kPairThreads);
}

// Launch as a programmatic dependent of the previous kernel on the stream
// (see wait_prerequisite).
template <class... KArgs, class... Args>
cudaError_t pdl_launch(void (*kern)(KArgs...), int grid, int threads, cudaStream_t st,
                       Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// f(dim, mode, log2 of the lanes a particle) with the compile-time constants
// of this cell list.
template <class F>
cudaError_t pair_dispatch(const CellList& cl, ab_op op, F&& f) {
    const int lanes_log2 = pair_lanes_log2(cl, op);
    auto with_split = [&](auto dim, auto mode) {
        switch (lanes_log2) {
            case 1: return f(dim, mode, std::integral_constant<int, 1>{});
            case 2: return f(dim, mode, std::integral_constant<int, 2>{});
            case 3: return f(dim, mode, std::integral_constant<int, 3>{});
            case 5: return f(dim, mode, std::integral_constant<int, 5>{});
            default: return f(dim, mode, std::integral_constant<int, 0>{});
        }
    };
    auto with_mode = [&](auto dim) {
        if (cl.g.general) return with_split(dim, std::integral_constant<int, kModeGeneral>{});
        if (cl.g.compact) return with_split(dim, std::integral_constant<int, kModeCompact>{});
        return with_split(dim, std::integral_constant<int, kModeFast>{});
    };
    return cl.g.dim == 3 ? with_mode(std::integral_constant<int, 3>{})
                         : with_mode(std::integral_constant<int, 2>{});
}

#define AB_PAIR_LAUNCH(...)                                                              \
    pair_dispatch(cl, op, [&](auto dim, auto mode, auto lanes) {                         \
        constexpr int DIM = decltype(dim)::value, MODE = decltype(mode)::value;          \
        constexpr int SL = decltype(lanes)::value;                                       \
        return pdl_launch(__VA_ARGS__, pair_blocks(cl, SL), kPairThreads, st, P, o);     \
    })

}  // namespace

}  // namespace ab
