// Dense kernel operator out = K(X, Y) W with K_ij = exp(-s |x_i - y_j|^2)
// and its adjoint (the RBF / Gaussian-process operators of paper Sec. 1 and
// Sec. 1.1; dense global operators, Sec. 2.2.2) on FP32 CUDA cores.
//
// One kernel, k_dense_own, serves the forward and every gradient.  Each
// thread owns I points (its rows) and walks a range of the other points,
// staged in shared memory and read as broadcasts; per pair it evaluates
// d = o - y, |d|^2 and K = 2^(-s log2e |d|^2) once and adds to
//   VAL   v_o[c] += K B[c]             (the product, or dW with roles swapped)
//   GRAD  S = sum_c A_o[c] B[c],  g_o += S K d,  e_o += S K |d|^2
//         (dX and ds, or dY with roles swapped)
// in registers.  VAL and GRAD together give dW and dY in one walk.
//
// Why this shape (65,536^2 pairs unless a size is given; the form before it
// was a 128 x 64 tile product through shared memory, always 64 columns wide,
// one block per 128 rows, and a separate scalar gradient kernel):
//  - The right-hand sides are compiled in powers of two (R), so one target
//    costs 8 FP32 operations a pair and not 7 + 64.
//  - Distances are formed for two rows at once and products for two columns
//    at once (f32x2: half the issue slots; the FP32 pipe itself runs 128
//    lane-operations a clock per SM either way).
//  - A broadcast shared load of 16 bytes takes about two clocks of the SM's
//    shared-memory pipe, so it has to feed many operations: I = 4 rows a
//    thread (2 where the gradient's registers leave no room).
//  - Few rows leave the chip idle, so the walk is split over the other
//    points as well (plan_split); the splits' partial sums are combined in a
//    fixed order by k_dense_combine, so results do not depend on timing.
//
// Bound: the FP32 pipe (7 + R operations a pair for values, 12 + R for
// gradients, 128 a clock per SM).  Measured against the tile form, forward /
// whole adjoint, us (and the forward's time at the pipe's rate):
//   65,536 x 65,536, 64 columns   16,129 / 67,786 -> 10,921 / 33,158  (8,038)
//   65,536 x 65,536,  1 column    16,042 / 66,625 ->  1,018 /  3,514    (906)
//   16,384 x 16,384, 32 columns    1,465 /  5,851 ->    371 /  1,147    (276)
//    5,001 x 12,345, 16 columns    1,102 /  2,783 ->     59 /    177     (37)
//    2,000 x 30,000,  1 column     2,649 /  4,479 ->     25 /     74     (13)
#include <cuda_runtime.h>
#include <stdint.h>

#include "ab_internal.cuh"

namespace ab {

namespace {

constexpr int kOwnThreads = 128;
constexpr float kLog2eD = 1.4426950408889634f;

__device__ __forceinline__ float ex2f(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Packed FP32 pairs: each half rounds exactly like the scalar operation.
__device__ __forceinline__ uint64_t f2p(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2u(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ uint64_t fsub2(uint64_t a, uint64_t b) {
    uint64_t d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool live) {
    const int sz = live ? 16 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void* src, bool live) {
    const int sz = live ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

struct OwnArgs {
    int64_t m, n;              // owned and other points
    const float4* O;           // owned points
    const float4* P;           // other points
    int nrhs;                  // columns of A and B
    const float* A;            // GRAD: weights of the owned points [m][nrhs]
    const float* B;            // weights of the other points [n][nrhs]
    float ns_log2e;            // -s log2(e)
    float gscale;              // GRAD: factor of the written gradient (-2 s)
    float* val;                // VAL: [m][nrhs], or the splits' partials [gridDim.y][m][nrhs]
    float4* grad;              // GRAD: [m], or partials [gridDim.y][m] (may be NULL)
    double* ds;                // GRAD: -sum e_o per block (may be NULL)
};

// R: columns a thread carries (a power of two); I: rows a thread owns (even).
// gridDim = (row blocks, splits of the other points, column groups of R).
template <int R, int I, bool VAL, bool GRAD, int OCC>
__global__ void __launch_bounds__(kOwnThreads, OCC)
k_dense_own(OwnArgs a) {
    static_assert(I % 2 == 0 && (R & (R - 1)) == 0, "rows in pairs, columns a power of two");
    constexpr int CH = R > 32 ? 64 : 128;     // points a stage
    // Points a turn of the loop, so that loads and exponentials of some run
    // under the products of others.  32 columns leave no registers for a
    // second point's products: values alone then evaluate the next point's K
    // under this point's products (PIPE).  16,384^2 pairs, forward / adjoint,
    // us, with 4, 2 (8 and 16 columns) and 1 (32) points a turn -> this:
    //   4 columns 107 / 350 -> 98 / 345     8: 147 / 496 -> 138 / 469
    //   16: 249 / 753 -> 225 / 704          32: 444 / 1,260 -> 405 / 1,226
    // (PIPE at 16 columns 227-235, more or fewer resident blocks no better.)
    constexpr int TURN = R >= 32 ? (GRAD ? 2 : 1) : R >= 2 ? 8 : 4;
    constexpr bool PIPE = VAL && !GRAD && R >= 32;
    constexpr int NP = I / 2;                 // row pairs
    constexpr int R2 = R > 1 ? R / 2 : 1;     // column pairs
    __shared__ __align__(16) float4 Ys[2][CH];
    __shared__ __align__(16) float Bs[2][CH * R];
    // lets the combining kernel be scheduled early (it waits for this grid)
    asm volatile("griddepcontrol.launch_dependents;");

    const int t = threadIdx.x;
    const int64_t row0 = (int64_t)blockIdx.x * (kOwnThreads * I) + t;
    const int c0 = blockIdx.z * R;
    const int nc = a.nrhs - c0 < R ? a.nrhs - c0 : R;
    const int64_t j_begin = a.n * blockIdx.y / gridDim.y;
    const int64_t j_end = a.n * (blockIdx.y + 1) / gridDim.y;

    // Aligned rows of whole float4s are copied, read and written 16 bytes at a
    // time: a warp's 4-byte accesses at a row's stride cost a sector each (16,384^2
    // pairs, forward / adjoint, us: 8 columns 138 / 471 -> 137 / 461, 16: 225 /
    // 705 -> 213 / 680, 32: 404 / 1,227 -> 371 / 1,147; 5,001 x 12,345 in 45
    // ranges with 16: 73 / 198 -> 62 / 183.  4 columns lose, 99 -> 102.)
    auto wide = [&](const float* q) { return a.nrhs % 4 == 0 && ((uintptr_t)q & 15u) == 0; };

    uint64_t ox[NP], oy[NP], oz[NP];   // owned points, rows (2p, 2p + 1) packed
    uint64_t av[GRAD ? I : 1][R2];     // GRAD: their weights (R = 1: in the low half)
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float4 o[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t row = row0 + (2 * p + u) * kOwnThreads;
            o[u] = row < a.m ? __ldg(a.O + row) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (GRAD && R >= 8 && wide(a.A)) {
#pragma unroll
                for (int c = 0; c < R2; c += 2) {
                    const float4 w = row < a.m && 2 * c < nc
                                         ? __ldg(reinterpret_cast<const float4*>(a.A + row * a.nrhs + 2 * c))
                                         : make_float4(0.f, 0.f, 0.f, 0.f);
                    av[2 * p + u][c] = f2p(w.x, w.y);
                    av[2 * p + u][c + 1 < R2 ? c + 1 : c] = f2p(w.z, w.w);
                }
            } else if (GRAD) {
#pragma unroll
                for (int c = 0; c < R2; ++c) {
                    const float* q = a.A + row * a.nrhs + 2 * c;
                    const float lo = row < a.m && 2 * c < nc ? __ldg(q) : 0.f;
                    const float hi = row < a.m && R > 1 && 2 * c + 1 < nc ? __ldg(q + 1) : 0.f;
                    av[2 * p + u][c] = f2p(lo, hi);
                }
            }
        }
        ox[p] = f2p(o[0].x, o[1].x);
        oy[p] = f2p(o[0].y, o[1].y);
        oz[p] = f2p(o[0].z, o[1].z);
    }
    // sums: VAL per row and column pair (R = 1: per row pair); GRAD per row pair
    uint64_t v[VAL ? (R > 1 ? I : NP) : 1][R2];
    uint64_t gx[NP], gy[NP], gz[NP], ge[NP];
#pragma unroll
    for (int q = 0; q < (VAL ? (R > 1 ? I : NP) : 1); ++q)
#pragma unroll
        for (int c = 0; c < R2; ++c) v[q][c] = 0ull;
#pragma unroll
    for (int p = 0; p < NP; ++p) gx[p] = gy[p] = gz[p] = ge[p] = 0ull;
    // GRAD: the sums over the stages before.  Four stages are summed by
    // themselves and added, so that a row's chain is 512 points and then their
    // number, not all points (unsplit walks, whole waves of row blocks: 20,000
    // equal terms were off by 2.9e-4, 77,824 x 10,000 with 64 columns and terms
    // of one sign by 9.4e-7 of their sum, rms, the tile form, two chains, by
    // 4.8e-7; this 4.5e-8).  Every stage folded, and in the same place: adjoint
    // of 16,384^2 with 4 columns 357 -> 366 us, this 362; 16 690 -> 687.
    uint64_t tx[NP], ty[NP], tz[NP], te[NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) tx[p] = ty[p] = tz[p] = te[p] = 0ull;
    int stages = 0;
    auto fold = [&] {
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            tx[p] = fadd2(tx[p], gx[p]);
            ty[p] = fadd2(ty[p], gy[p]);
            tz[p] = fadd2(tz[p], gz[p]);
            te[p] = fadd2(te[p], ge[p]);
            gx[p] = gy[p] = gz[p] = ge[p] = 0ull;
        }
    };

    auto stage = [&](int64_t j0, int b) {
        for (int q = t; q < CH; q += kOwnThreads) {
            const bool live = j0 + q < j_end;
            cp_async16((uint32_t)__cvta_generic_to_shared(&Ys[b][q]), a.P + (live ? j0 + q : 0), live);
        }
        if (R >= 8 && wide(a.B)) {
#pragma unroll 4
            for (int e = t; e < CH * R / 4; e += kOwnThreads) {
                const int jj = e / (R / 4 ? R / 4 : 1), c = e % (R / 4 ? R / 4 : 1) * 4;
                const bool live = j0 + jj < j_end && c < nc;
                cp_async16((uint32_t)__cvta_generic_to_shared(&Bs[b][4 * e]),
                           a.B + (live ? (j0 + jj) * a.nrhs + c0 + c : 0), live);
            }
            cp_async_commit();
            return;
        }
#pragma unroll 4
        for (int k = 0; k < CH * R / kOwnThreads; ++k) {
            const int e = k * kOwnThreads + t;
            const int jj = e / R, c = e % R;
            const bool live = j0 + jj < j_end && c < nc;
            cp_async4((uint32_t)__cvta_generic_to_shared(&Bs[b][e]),
                      a.B + (live ? (j0 + jj) * a.nrhs + c0 + c : 0), live);
        }
        cp_async_commit();
    };

    const uint64_t ns2 = f2p(a.ns_log2e, a.ns_log2e);
    int b = 0;
    if (j_begin < j_end) stage(j_begin, 0);
    for (int64_t j0 = j_begin; j0 < j_end; j0 += CH, b ^= 1) {
        cp_async_wait_all();
        __syncthreads();       // stage b is complete, and the other one fully read
        if (j0 + CH < j_end) stage(j0 + CH, b ^ 1);
        const int cnt = (int)(j_end - j0 < CH ? j_end - j0 : CH);
        const float4* __restrict__ Yb = Ys[b];
        const float* __restrict__ Bb = Bs[b];
        if constexpr (PIPE) {
            auto kernel = [&](int j, uint64_t (&k)[NP]) {
                const float4 y = Yb[j];
                const uint64_t yx = f2p(y.x, y.x), yy = f2p(y.y, y.y), yz = f2p(y.z, y.z);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const uint64_t dx = fsub2(ox[p], yx), dy = fsub2(oy[p], yy), dz = fsub2(oz[p], yz);
                    const uint64_t d2 = ffma2(dz, dz, ffma2(dy, dy, fmul2(dx, dx)));
                    float e0, e1;
                    f2u(fmul2(d2, ns2), e0, e1);
                    k[p] = f2p(ex2f(e0), ex2f(e1));
                }
            };
            uint64_t k2[NP];
            kernel(0, k2);
#pragma unroll 1
            for (int j = 0; j < cnt; ++j) {
                uint64_t next[NP];
                kernel(j + 1 < CH ? j + 1 : 0, next);   // the last one's is not used
#pragma unroll
                for (int c = 0; c < R2; c += 2) {
                    const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(Bb + j * R + 2 * c);
#pragma unroll
                    for (int p = 0; p < NP; ++p) {
                        float k0, k1;
                        f2u(k2[p], k0, k1);
                        const uint64_t kk0 = f2p(k0, k0), kk1 = f2p(k1, k1);
                        v[2 * p][c] = ffma2(kk0, w.x, v[2 * p][c]);
                        v[2 * p + 1][c] = ffma2(kk1, w.x, v[2 * p + 1][c]);
                        v[2 * p][c + 1] = ffma2(kk0, w.y, v[2 * p][c + 1]);
                        v[2 * p + 1][c + 1] = ffma2(kk1, w.y, v[2 * p + 1][c + 1]);
                    }
                }
#pragma unroll
                for (int p = 0; p < NP; ++p) k2[p] = next[p];
            }
            continue;
        }
#pragma unroll TURN
        for (int j = 0; j < cnt; ++j) {
            const float4 y = Yb[j];
            const uint64_t yx = f2p(y.x, y.x), yy = f2p(y.y, y.y), yz = f2p(y.z, y.z);
            uint64_t B2[R2];
            if (R == 1) {
                B2[0] = f2p(Bb[j], Bb[j]);
            } else if (R == 2) {
                B2[0] = *reinterpret_cast<const uint64_t*>(Bb + j * R);
            } else {
#pragma unroll
                for (int c = 0; c < R2; c += 2) {
                    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(Bb + j * R + 2 * c);
                    B2[c] = q.x;
                    B2[c + 1 < R2 ? c + 1 : c] = q.y;
                }
            }
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                const uint64_t dx = fsub2(ox[p], yx), dy = fsub2(oy[p], yy), dz = fsub2(oz[p], yz);
                const uint64_t d2 = ffma2(dz, dz, ffma2(dy, dy, fmul2(dx, dx)));
                float e0, e1;
                f2u(fmul2(d2, ns2), e0, e1);
                const float k0 = ex2f(e0), k1 = ex2f(e1);
                const uint64_t k2 = f2p(k0, k1);
                if (VAL) {
                    if (R == 1) {
                        v[p][0] = ffma2(k2, B2[0], v[p][0]);
                    } else {
                        const uint64_t kk0 = f2p(k0, k0), kk1 = f2p(k1, k1);
                        constexpr int q0 = 2;
#pragma unroll
                        for (int c = 0; c < R2; ++c) {
                            v[R > 1 ? q0 * p : 0][c] = ffma2(kk0, B2[c], v[R > 1 ? q0 * p : 0][c]);
                            v[R > 1 ? q0 * p + 1 : 0][c] = ffma2(kk1, B2[c], v[R > 1 ? q0 * p + 1 : 0][c]);
                        }
                    }
                }
                if (GRAD) {
                    uint64_t S2;
                    if (R == 1) {
                        float w0, w1, a0, a1, z;
                        f2u(B2[0], w0, w1);
                        f2u(av[GRAD ? 2 * p : 0][0], a0, z);
                        f2u(av[GRAD ? 2 * p + 1 : 0][0], a1, z);
                        S2 = fmul2(f2p(a0, a1), f2p(w0, w1));
                    } else {
                        uint64_t s0 = 0ull, s1 = 0ull;
#pragma unroll
                        for (int c = 0; c < R2; ++c) {
                            s0 = ffma2(av[GRAD ? 2 * p : 0][c], B2[c], s0);
                            s1 = ffma2(av[GRAD ? 2 * p + 1 : 0][c], B2[c], s1);
                        }
                        float l0, h0, l1, h1;
                        f2u(s0, l0, h0);
                        f2u(s1, l1, h1);
                        S2 = f2p(l0 + h0, l1 + h1);
                    }
                    const uint64_t A2 = fmul2(S2, k2);
                    gx[p] = ffma2(A2, dx, gx[p]);
                    gy[p] = ffma2(A2, dy, gy[p]);
                    gz[p] = ffma2(A2, dz, gz[p]);
                    ge[p] = ffma2(A2, d2, ge[p]);
                }
            }
        }
        if constexpr (GRAD) {
            if ((++stages & 3) == 0) fold();
        }
    }
    if constexpr (GRAD) fold();

    double dsum = 0.0;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        float x[2], y[2], z[2], e[2], w[2];
        f2u(GRAD ? tx[p] : gx[p], x[0], x[1]);
        f2u(GRAD ? ty[p] : gy[p], y[0], y[1]);
        f2u(GRAD ? tz[p] : gz[p], z[0], z[1]);
        f2u(GRAD ? te[p] : ge[p], e[0], e[1]);
        f2u(v[VAL && R == 1 ? p : 0][0], w[0], w[1]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int64_t row = row0 + (2 * p + u) * kOwnThreads;
            if (row >= a.m) continue;
            if (VAL) {
                float* q = a.val + ((int64_t)blockIdx.y * a.m + row) * a.nrhs + c0;
                if (R == 1) {
                    q[0] = w[u];
                } else if (R >= 8 && wide(a.val)) {
#pragma unroll
                    for (int c = 0; c < R2; c += 2) {
                        float4 f;
                        f2u(v[R > 1 ? 2 * p + u : 0][c], f.x, f.y);
                        f2u(v[R > 1 ? 2 * p + u : 0][c + 1 < R2 ? c + 1 : c], f.z, f.w);
                        if (2 * c < nc) *reinterpret_cast<float4*>(q + 2 * c) = f;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < R2; ++c) {
                        float lo, hi;
                        f2u(v[R > 1 ? 2 * p + u : 0][c], lo, hi);
                        if (2 * c < nc) q[2 * c] = lo;
                        if (2 * c + 1 < nc) q[2 * c + 1] = hi;
                    }
                }
            }
            if (GRAD) {
                if (a.grad)
                    a.grad[(int64_t)blockIdx.y * a.m + row] =
                        make_float4(a.gscale * x[u], a.gscale * y[u], a.gscale * z[u], 0.f);
                dsum -= (double)e[u];
            }
        }
    }
    if (GRAD && a.ds) {   // FP64 block sum in a fixed order
        __shared__ double s_red[kOwnThreads / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) dsum += __shfl_down_sync(0xffffffffu, dsum, o);
        if ((t & 31) == 0) s_red[t >> 5] = dsum;
        __syncthreads();
        if (t == 0) {
            double tot = 0.0;
#pragma unroll
            for (int q = 0; q < kOwnThreads / 32; ++q) tot += s_red[q];
            a.ds[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
        }
    }
}

// Sum of splits partials `stride` apart, in their order, N loads in flight (the
// last batch loads its end again rather than one by one).
template <int N>
__device__ __forceinline__ float sum_splits(const float* __restrict__ p, int splits, int64_t stride) {
    float s = 0.f;
#pragma unroll 1
    for (int q0 = 0; q0 < splits; q0 += N) {
        float x[N];
#pragma unroll
        for (int u = 0; u < N; ++u) x[u] = __ldcg(p + min(q0 + u, splits - 1) * stride);
#pragma unroll
        for (int u = 0; u < N; ++u) s += q0 + u < splits ? x[u] : 0.f;
    }
    return s;
}

// Sums of the splits' partials, in the order of the splits: `vals` floats and
// `grads` float4 (either may be 0).  Few rows have many splits and then wait
// for the loads alone, so many are in flight at a time (against 8 and the rest
// one by one, us, product / adjoint: 100 x 60,000 points 26.7 / 55 -> 20.6 / 39,
// 2,000 x 30,000 28.7 / 80 -> 24.7 / 74, 300 x 4,000 with 8 columns 12.4 / 29 ->
// 10.3 / 23).
__global__ void __launch_bounds__(256)
k_dense_combine(int splits, int64_t vals, const float* __restrict__ pv, float* __restrict__ val,
                int64_t grads, const float4* __restrict__ pg, float4* __restrict__ grad) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e < vals) {
        val[e] = splits > 16  ? sum_splits<32>(pv + e, splits, vals)
                 : splits > 8 ? sum_splits<16>(pv + e, splits, vals)
                              : sum_splits<8>(pv + e, splits, vals);
    } else if (e - vals < grads) {
        constexpr int N = 16;
        const int64_t r = e - vals;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int q0 = 0; q0 < splits; q0 += N) {
            float4 g[N];
#pragma unroll
            for (int u = 0; u < N; ++u) g[u] = __ldcg(pg + min(q0 + u, splits - 1) * grads + r);
#pragma unroll
            for (int u = 0; u < N; ++u) {
                const bool in = q0 + u < splits;
                s.x += in ? g[u].x : 0.f;
                s.y += in ? g[u].y : 0.f;
                s.z += in ? g[u].z : 0.f;
            }
        }
        grad[r] = s;
    }
}

// Columns a thread carries, rows it owns and blocks per SM for a pass.
// ORDERED values (the solve's product, whose iteration count follows the last
// bits) keep one chain of FMAs per output over the points in increasing
// index: no split, two rows a thread, and fewer columns a thread where that
// brings more SMs to work (K is then evaluated once per column group).
struct OwnShape {
    int R, I, occ;
};

// VAL alone: the cheapest power of two by its operations per pair (7 for the
// distance and the exponent, one per column), counting the columns padded.
// A gradient needs all columns in one thread: the next power of two.
OwnShape own_shape(int nrhs, bool val, bool grad) {
    if (!grad) {
        int best = 32, cost = 1 << 30;
        for (int R = 1; R <= 32; R *= 2) {
            const int c = ((nrhs + R - 1) / R) * (7 + R);
            if (c < cost) {
                cost = c;
                best = R;
            }
        }
        return {best, 4, best >= 32 ? 2 : best >= 16 ? 3 : 4};
    }
    int R = 1;
    while (R < nrhs) R *= 2;
    (void)val;
    return {R, 2, R >= 32 ? 2 : R >= 16 ? 3 : 4};
}

OwnShape ordered_shape(int64_t m, int nrhs) {
    OwnShape best = {1, 2, 4};
    int64_t cost = INT64_MAX;
    for (int R = 1; R <= 32; R *= 2) {
        const int groups = (nrhs + R - 1) / R;
        const int64_t blocks = (m + 2 * kOwnThreads - 1) / (2 * kOwnThreads) * groups;
        // a block alone on its SM runs at the latency of its FMAs, about the
        // time that two blocks take together
        int64_t per_sm = (blocks + num_sms() - 1) / num_sms();
        if (per_sm < 2) per_sm = 2;
        const int64_t c = per_sm * (7 + R);
        if (c < cost) {
            cost = c;
            best = {R, 2, R >= 32 ? 2 : R >= 16 ? 3 : 4};
        }
        if (R >= nrhs) break;
    }
    return best;
}

// Splits of the n other points: the work of a block is its points plus about
// 64 points' worth of start and write-out, and blocks run in waves of the
// resident ones; the number of splits with the least time in that model whose
// partial sums (split_bytes each) take at most kMaxPartBytes.  The context keeps
// them, and many rows gain only the last wave by them: 200,000^2 points with 64
// columns took 12 splits and 586 MB, now 3 and 146 MB (100.0 -> 103.8 ms), 10^6
// rows 7 and 1.7 GB for 1%, now 1.  65,536^2 keeps its 13 (208 MB, 10.9 ms).
constexpr int64_t kMaxPartBytes = int64_t(224) << 20;

int plan_split(int64_t blocks, int64_t n, int occ, int64_t split_bytes) {
    const int64_t resident = (int64_t)occ * num_sms();
    int64_t most = (n + 63) / 64;
    if (most > 256) most = 256;
    if (split_bytes > 0 && most > kMaxPartBytes / split_bytes) most = kMaxPartBytes / split_bytes;
    int64_t best = 1, cost = INT64_MAX;
    for (int64_t s = 1; s <= most; ++s) {
        const int64_t waves = (blocks * s + resident - 1) / resident;
        const int64_t c = waves * ((n + s - 1) / s + 64) + s / 4;
        if (c < cost) {
            cost = c;
            best = s;
        }
    }
    return (int)best;
}

struct OwnPlan {
    OwnShape sh;
    int64_t blocks;   // row blocks
    int groups;       // column groups
    int splits;
};

OwnPlan own_plan(int64_t m, int64_t n, int nrhs, bool val, bool grad, bool may_split) {
    OwnPlan p;
    p.sh = own_shape(nrhs, val, grad);
    const int64_t rows = (int64_t)kOwnThreads * p.sh.I;
    p.blocks = (m + rows - 1) / rows;
    p.groups = grad ? 1 : (nrhs + p.sh.R - 1) / p.sh.R;
    const int64_t split_bytes = m * ((val ? (int64_t)nrhs * 4 : 0) + (grad ? 16 : 0));
    p.splits = may_split ? plan_split(p.blocks * p.groups, n, p.sh.occ, split_bytes) : 1;
    return p;
}

size_t own_bytes(const OwnPlan& p, int64_t m, int nrhs, bool val, bool grad) {
    if (p.splits <= 1) return 0;
    return (size_t)p.splits * m * ((val ? (size_t)nrhs * 4 : 0) + (grad ? 16 : 0)) + 32;
}

template <int R, bool VAL, bool GRAD>
void own_launch(const OwnPlan& p, const OwnArgs& a, cudaStream_t st) {
    constexpr int OCC = R >= 32 ? 2 : R >= 16 ? 3 : 4;
    const dim3 grid((unsigned)p.blocks, (unsigned)p.splits, (unsigned)p.groups);
    if constexpr (!GRAD) {
        if (p.sh.I == 4) {
            k_dense_own<R, 4, VAL, GRAD, OCC><<<grid, kOwnThreads, 0, st>>>(a);
            return;
        }
    }
    k_dense_own<R, 2, VAL, GRAD, OCC><<<grid, kOwnThreads, 0, st>>>(a);
}

template <bool VAL, bool GRAD>
cudaError_t own_dispatch(const OwnPlan& p, const OwnArgs& a, cudaStream_t st) {
    switch (p.sh.R) {
        case 1: own_launch<1, VAL, GRAD>(p, a, st); break;
        case 2: own_launch<2, VAL, GRAD>(p, a, st); break;
        case 4: own_launch<4, VAL, GRAD>(p, a, st); break;
        case 8: own_launch<8, VAL, GRAD>(p, a, st); break;
        case 16: own_launch<16, VAL, GRAD>(p, a, st); break;
        case 32: own_launch<32, VAL, GRAD>(p, a, st); break;
        case 64:
            if constexpr (GRAD && !VAL) {
                own_launch<64, VAL, GRAD>(p, a, st);
                break;
            }
            return cudaErrorInvalidValue;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// One pass: values and / or gradients of the m owned points.  ws: the
// splits' partials (own_bytes), or NULL to walk unsplit.  ds: per-block
// partials, *ds_count of them.
cudaError_t own_pass(int64_t m, int64_t n, const float4* O, const float4* P, int nrhs,
                     const float* A, const float* B, float s, float* val, bool want_grad,
                     float4* grad, double* ds, int* ds_count, void* ws, cudaStream_t st) {
    const bool want_val = val != nullptr;
    const OwnPlan p = own_plan(m, n, nrhs, want_val, want_grad, ws != nullptr);
    OwnArgs a;
    a.m = m;
    a.n = n;
    a.O = O;
    a.P = P;
    a.nrhs = nrhs;
    a.A = A;
    a.B = B;
    a.ns_log2e = -s * kLog2eD;
    a.gscale = -2.f * s;
    a.val = val;
    a.grad = grad;
    a.ds = ds;
    float4* pg = (float4*)ws;   // gradients first: 16-byte aligned
    const int64_t ng = grad ? m : 0, nv = want_val ? m * nrhs : 0;
    float* pv = (float*)(pg + (p.splits > 1 ? p.splits * ng : 0));
    if (p.splits > 1) {
        if (want_val) a.val = pv;
        if (grad) a.grad = pg;
    }
    cudaError_t e = want_val ? (want_grad ? own_dispatch<true, true>(p, a, st)
                                          : own_dispatch<true, false>(p, a, st))
                             : own_dispatch<false, true>(p, a, st);
    if (e != cudaSuccess) return e;
    if (ds_count) *ds_count = (int)(p.blocks * p.splits);
    if (p.splits > 1 && nv + ng > 0)
        e = launch_dense_combine(p.splits, nv, pv, val, ng, pg, grad, st);
    return e;
}

// dW and dY share a walk while both fit a thread's registers.
constexpr int kFusedRhs = 32;

}  // namespace

cudaError_t launch_dense_combine(int splits, int64_t vals, const float* pv, float* val, int64_t grads,
                                 const float4* pg, float4* grad, cudaStream_t st) {
    // programmatic dependent launch: scheduled while the walk runs, waits in
    // griddepcontrol.wait for its writes
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((vals + grads + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_dense_combine, splits, vals, pv, val, grads, pg, grad);
}

size_t dense_fwd_workspace_bytes(int64_t m, int64_t n, int nrhs) {
    if (m <= 0 || n <= 0) return 0;
    return own_bytes(own_plan(m, n, nrhs, true, false, true), m, nrhs, true, false);
}

size_t dense_bwd_workspace_bytes(int64_t m, int64_t n, int nrhs, bool dW, bool dX, bool dY, bool ds) {
    size_t need = 0;
    auto take = [&](int64_t rows, int64_t other, bool v, bool g) {
        if (rows <= 0 || other <= 0) return;
        const size_t b = own_bytes(own_plan(rows, other, nrhs, v, g, true), rows, nrhs, v, g);
        if (b > need) need = b;
    };
    if (dX || ds) take(m, n, false, true);
    if (dW && dY && nrhs <= kFusedRhs) {
        take(n, m, true, true);
    } else {
        if (dW) take(n, m, true, false);
        if (dY) take(n, m, false, true);
    }
    return need;
}

size_t dense_partial_capacity(int64_t m, int64_t n, int nrhs) {
    if (m <= 0 || n <= 0) return 1;
    const OwnPlan p = own_plan(m, n, nrhs, false, true, true);
    return (size_t)(p.blocks * p.splits);
}

cudaError_t launch_dense_fwd(int64_t m, int64_t n, const float4* X, const float4* Y,
                             int nrhs, const float* W, float s, float* out, void* ws,
                             cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    if (n <= 0) return cudaMemsetAsync(out, 0, (size_t)m * nrhs * sizeof(float), st);
    return own_pass(m, n, X, Y, nrhs, nullptr, W, s, out, false, nullptr, nullptr, nullptr, ws, st);
}

cudaError_t launch_dense_fwd_ordered(int64_t m, int64_t n, const float4* X, const float4* Y,
                                     int nrhs, const float* W, float s, float* out,
                                     cudaStream_t st) {
    if (m <= 0) return cudaSuccess;
    if (n <= 0) return cudaMemsetAsync(out, 0, (size_t)m * nrhs * sizeof(float), st);
    OwnPlan p;
    p.sh = ordered_shape(m, nrhs);
    p.blocks = (m + kOwnThreads * p.sh.I - 1) / (kOwnThreads * p.sh.I);
    p.groups = (nrhs + p.sh.R - 1) / p.sh.R;
    p.splits = 1;
    OwnArgs a = {};
    a.m = m;
    a.n = n;
    a.O = X;
    a.P = Y;
    a.nrhs = nrhs;
    a.B = W;
    a.ns_log2e = -s * kLog2eD;
    a.val = out;
    return own_dispatch<true, false>(p, a, st);
}

cudaError_t launch_dense_bwd(int64_t m, int64_t n, const float4* X, const float4* Y,
                             int nrhs, const float* W, float s, const float* G, float* dW,
                             float4* dX, float4* dY, double* partial, int* partial_count,
                             void* ws, cudaStream_t st) {
    cudaError_t e = cudaSuccess;
    *partial_count = 0;
    if (n > 0 && m <= 0) {
        if (dW && (e = cudaMemsetAsync(dW, 0, (size_t)n * nrhs * sizeof(float), st)) != cudaSuccess) return e;
        if (dY && (e = cudaMemsetAsync(dY, 0, (size_t)n * sizeof(float4), st)) != cudaSuccess) return e;
        return e;
    }
    if (m > 0 && n <= 0)
        return dX ? cudaMemsetAsync(dX, 0, (size_t)m * sizeof(float4), st) : cudaSuccess;
    if (m <= 0) return cudaSuccess;
    if (dX || partial) {
        e = own_pass(m, n, X, Y, nrhs, G, W, s, nullptr, true, dX, partial, partial_count, ws, st);
        if (e != cudaSuccess) return e;
    }
    // K(X, Y)^T = K(Y, X): the columns own, the rows are walked
    if (dW && dY && nrhs <= kFusedRhs)
        return own_pass(n, m, Y, X, nrhs, W, G, s, dW, true, dY, nullptr, nullptr, ws, st);
    if (dW) {
        e = own_pass(n, m, Y, X, nrhs, nullptr, G, s, dW, false, nullptr, nullptr, nullptr, ws, st);
        if (e != cudaSuccess) return e;
    }
    if (dY) e = own_pass(n, m, Y, X, nrhs, W, G, s, nullptr, true, dY, nullptr, nullptr, ws, st);
    return e;
}

}  // namespace ab
