// Kernel kernels of the conjugate-gradient solve of (K(X, X) + sigma^2 I) W = B
// (the linear system of RBF interpolation with a nugget and of the
// Gaussian-process posterior mean, paper Sec. 1.1; Hestenes and Stiefel's
// method, one independent CG per right-hand side).
//
// Vectors are float32 [n][nrhs] row-major.  Every inner product is a per-
// column FP64 sum: a block of 4 x 64 threads covers 64 columns and a range of
// rows, reduces its rows in shared memory, and writes one partial per
// (block, column); a second kernel adds the partials of each column in a
// fixed order, so the result is the same on every run.  The step lengths
// alpha = (r.r) / (p.Ap) and beta = (r'.r') / (r.r) are formed on the device
// in FP64; a column whose residual has reached tol ||b|| is frozen (alpha =
// beta = 0, p = 0).  A p = K p + sigma^2 p is never stored: the kernels that
// need it take K p and p.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <vector>

#include "ab_internal.cuh"

namespace ab {

namespace {

constexpr int kCols = 64;       // columns per block (threadIdx.x)
constexpr int kRowLanes = 4;    // row lanes per block (threadIdx.y)

// Per-column scalars of the iteration (device, FP64).
struct Col {
    double bb;      // b.b
    double rs;      // r.r of the current residual
    double pap;     // p.(K p + sigma^2 p)
    double rs_new;  // r.r after the update
    double beta;    // rs_new / rs
    int active;     // 1 while ||r|| > tol ||b||
    int pad;
};

__device__ __forceinline__ void row_range(int64_t n, int64_t& r0, int64_t& r1) {
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    r0 = per * blockIdx.x;
    r1 = r0 + per < n ? r0 + per : n;
}

// Reduce v over threadIdx.y and store partial[blockIdx.x][c].
__device__ __forceinline__ void col_partial(double v, int c, int nrhs, double* partial) {
    __shared__ double s[kRowLanes][kCols];
    s[threadIdx.y][threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.y == 0 && c < nrhs) {
        double t = 0.0;
#pragma unroll
        for (int q = 0; q < kRowLanes; ++q) t += s[q][threadIdx.x];
        partial[(int64_t)blockIdx.x * nrhs + c] = t;
    }
}

// The step kernels are programmatic dependent launches of the kernel before
// them: scheduled while it finishes, they wait here for its writes, and read
// what it wrote from L2 (col too, which k_solve_finish writes while the next
// one may already be resident).
__device__ __forceinline__ void solve_dependent() {
    asm volatile("griddepcontrol.launch_dependents;");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// R = B, P = B, W = 0; partial of b.b
__global__ void __launch_bounds__(kCols * kRowLanes)
k_solve_init(int64_t n, int nrhs, const float* __restrict__ B, float* __restrict__ R,
             float* __restrict__ P, float* __restrict__ W, double* __restrict__ partial) {
    const int c = blockIdx.y * kCols + threadIdx.x;
    int64_t r0, r1;
    row_range(n, r0, r1);
    double acc = 0.0;
    if (c < nrhs) {
        for (int64_t i = r0 + threadIdx.y; i < r1; i += kRowLanes) {
            const int64_t e = i * nrhs + c;
            const float b = __ldg(B + e);
            R[e] = b;
            P[e] = b;
            W[e] = 0.0f;
            acc += (double)b * b;
        }
    }
    col_partial(acc, c, nrhs, partial);
}

// partial of p.(q + sigma^2 p), q = K p
__global__ void __launch_bounds__(kCols * kRowLanes)
k_solve_pap(int64_t n, int nrhs, const float* __restrict__ P, const float* __restrict__ Q,
            float sigma2, double* __restrict__ partial, int* __restrict__ n_active) {
    solve_dependent();
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0 && threadIdx.y == 0) *n_active = 0;
    const int c = blockIdx.y * kCols + threadIdx.x;
    int64_t r0, r1;
    row_range(n, r0, r1);
    double acc = 0.0;
    if (c < nrhs) {
        for (int64_t i = r0 + threadIdx.y; i < r1; i += kRowLanes) {
            const int64_t e = i * nrhs + c;
            const double p = __ldcg(P + e);
            acc += p * ((double)__ldcg(Q + e) + (double)sigma2 * p);
        }
    }
    col_partial(acc, c, nrhs, partial);
}

// W += alpha p, R -= alpha (q + sigma^2 p); partial of the new r.r
__global__ void __launch_bounds__(kCols * kRowLanes)
k_solve_update(int64_t n, int nrhs, const float* __restrict__ P, const float* __restrict__ Q,
               float sigma2, const Col* col, float* __restrict__ R,
               float* __restrict__ W, double* __restrict__ partial) {
    solve_dependent();
    const int c = blockIdx.y * kCols + threadIdx.x;
    int64_t r0, r1;
    row_range(n, r0, r1);
    double acc = 0.0;
    if (c < nrhs) {
        const double rs = __ldcg(&col[c].rs), pap = __ldcg(&col[c].pap);
        const float alpha = (__ldcg(&col[c].active) && pap > 0.0) ? (float)(rs / pap) : 0.0f;
        for (int64_t i = r0 + threadIdx.y; i < r1; i += kRowLanes) {
            const int64_t e = i * nrhs + c;
            const float p = __ldcg(P + e);
            const float ap = fmaf(sigma2, p, __ldcg(Q + e));
            W[e] = fmaf(alpha, p, __ldcg(W + e));
            const float r = fmaf(-alpha, ap, __ldcg(R + e));
            R[e] = r;
            acc += (double)r * r;
        }
    }
    col_partial(acc, c, nrhs, partial);
}

// P = R + beta P (frozen columns: P = 0)
__global__ void __launch_bounds__(kCols * kRowLanes)
k_solve_dir(int64_t n, int nrhs, const float* __restrict__ R, const Col* col,
            float* __restrict__ P) {
    solve_dependent();
    const int c = blockIdx.y * kCols + threadIdx.x;
    int64_t r0, r1;
    row_range(n, r0, r1);
    if (c >= nrhs) return;
    const int active = __ldcg(&col[c].active);
    const float beta = (float)__ldcg(&col[c].beta);
    for (int64_t i = r0 + threadIdx.y; i < r1; i += kRowLanes) {
        const int64_t e = i * nrhs + c;
        P[e] = active ? fmaf(beta, __ldcg(P + e), __ldcg(R + e)) : 0.0f;
    }
}

// Column sum of the partials in a fixed order, then the scalar step for
// what = 0: b.b (initialise), 1: p.Ap, 2: r'.r' (beta, activity, counts).  One
// warp and block a column: FP64 additions take an SM's pipe for 16 clocks and
// more, and all columns on one SM took longer than the rest of a step.
__global__ void __launch_bounds__(32)
k_solve_finish(const double* __restrict__ partial, int blocks, int nrhs, int what, double tol2,
               Col* col, int* __restrict__ n_active) {
    solve_dependent();
    const int c = blockIdx.x, lane = threadIdx.x;
    double t = 0.0;
    for (int b = lane; b < blocks; b += 32) t += __ldcg(partial + (int64_t)b * nrhs + c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane != 0) return;
    Col k;
    k.bb = __ldcg(&col[c].bb);
    k.rs = __ldcg(&col[c].rs);
    k.pap = __ldcg(&col[c].pap);
    k.rs_new = __ldcg(&col[c].rs_new);
    k.beta = __ldcg(&col[c].beta);
    k.active = __ldcg(&col[c].active);
    k.pad = 0;
    if (what == 0) {
        k.bb = t;
        k.rs = t;
        k.pap = 0.0;
        k.rs_new = t;
        k.beta = 0.0;
        k.active = t > 0.0;
    } else if (what == 1) {
        k.pap = t;
    } else {
        k.rs_new = t;
        if (k.active) {
            k.beta = k.rs > 0.0 ? t / k.rs : 0.0;
            k.rs = t;
            k.active = t > tol2 * k.bb;
        } else {
            k.beta = 0.0;
        }
    }
    col[c] = k;
    if (what != 1 && k.active) atomicAdd(n_active, 1);
}

// ---------------------------------------------------------------------------
// The whole iteration in one cooperative launch, for FP32 systems of few
// right-hand sides (run_solve_coop).
//
// The product keeps the order of the plain one: a row's sum is one chain of
// FMAs over the points in increasing index.  The number of iterations, which
// callers see, depends on the last bits of q = K p (two orders of the same sum
// differ by one iteration in about one system of ten at tol 1e-4), so a split
// sum would change it.  A chain of n FMAs takes 4 n clocks however many
// threads there are, so everything else is kept off its path:
//   - K is evaluated once a call into a slab per block ([n / 4][rows][4
//     points]; n = 4096: 64 MB, which stays in L2), not once an iteration.
//   - Consumer warps hold one row a lane, all its columns in that lane, with
//     r, p, w and q in registers, and run the chains from shared memory.
//     They are warps 3 mod 4, alone on their scheduler.
//   - The other 12 warps stream the slab through a ring of three tiles
//     (cp.async, two tiles ahead, through the reductions as well) and form
//     the direction p of the next tile's points.
//   - Two all-reductions an iteration, p.Ap and r.r, are also its grid
//     barriers.  Each block pushes its sum with an epoch, in one 16-byte
//     word, into every block's mailbox and polls its own, so nothing contends
//     and nothing needs a fence; the sums are added in the same order
//     everywhere, so all blocks hold the same step lengths.
//   - The owner of a row publishes {r, p, epoch} in one 16-byte word, and
//     producers form p_j = r_j + beta p_j from it: the new direction costs no
//     barrier.  The word is rewritten only after the next p.Ap reduction,
//     which every block enters once it has read all words.
//
// Bound: the chain's latency (n = 4096: 16,384 clocks, 8.4 us an iteration)
// and the two reductions.  The form it replaces launched seven kernels an
// iteration on 16-32 blocks, padded one column to 64 and waited on the host
// each time.  n = 4096, one column, tol 1e-4, 69 iterations: 32.4 ms ->
// 1.57 ms, W and the iteration count bit for bit.  Of an iteration's 22.7
// us the chains take 17.5: 8.3 clocks a point beside the slab's copies (6.6
// without them, 5.1 with nothing else on the SM).  Measured on the way: K
// evaluated anew each iteration by the 12 warps 29 us an iteration (they, not
// the chain, set the pace), atomic barriers with fences about 9,000 clocks a
// reduction.
// ---------------------------------------------------------------------------
constexpr int kCoopT = 512;         // threads a block
constexpr int kCoopProd = 384;      // producers among them
constexpr int kCoopMaxGroups = 2;   // consumer warps, at most
constexpr int kCoopMaxCols = 4;
constexpr int kCoopMaxBlocks = 256;
constexpr long long kSolveWaitNs = 1000000000ll;

struct CoopResult {
    int iters;
    int done;        // 1 once block 0 has come to its end
    int failed;      // 1 if a wait of any block ran out
    int pad;
    double worst;    // largest r.r / b.b
};

// 16 bytes written and read at once: a value and the step it belongs to.
struct __align__(16) CoopWord {
    uint64_t value, epoch;
};

struct CoopSolve {
    int64_t n;
    int rows;                  // rows a block owns (the last block may own fewer)
    int groups;                // consumer warps: rows / 32, rounded up
    const float4* X;
    const float* B;
    float ns_log2e, sigma2;
    double tol2;
    int max_iter;
    float* W;                  // [n][nrhs]
    CoopWord* rp;              // [n][nrhs]: {r, p}; epochs 0 at launch
    CoopWord* mail;            // [2][nrhs][to][from]: partial sums; epochs 0 at launch
    float* slab;               // [blocks][n4 / 4][rows][4]
    CoopResult* result;
    long long limit_ns;        // testing: of each wait
    int skip_block;            // testing: this block takes no part
};

__device__ __forceinline__ float ex2_solve(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void word_store(CoopWord* s, uint64_t value, uint64_t epoch) {
    asm volatile(
        "{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\t"
        "st.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(s),
        "l"(value), "l"(epoch)
        : "memory");
}
__device__ __forceinline__ void word_load(const CoopWord* s, uint64_t& value, uint64_t& epoch) {
    asm volatile(
        "{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\t"
        "mov.b128 {%0, %1}, q;\n\t}"
        : "=l"(value), "=l"(epoch)
        : "l"(s)
        : "memory");
}
// A warp's wait for words of this epoch, one a live lane, for at most the time
// limit (*dead: an earlier wait of the block ran out; then not at all).  The
// loop's exit is the warp's vote: lanes leaving one by one would leave the
// warp split behind it (7.1 instead of 9.5 us an iteration at n = 500).
__device__ __forceinline__ bool word_wait(const CoopWord* s, bool live, uint64_t epoch, uint64_t& value,
                                          volatile int* dead, long long limit_ns) {
    long long t0 = 0;
    value = 0ull;
    for (int spin = 0;; ++spin) {
        uint64_t e = epoch;
        if (live) word_load(s, value, e);
        if (__all_sync(0xffffffffu, e == epoch)) return true;
        if ((spin & 63) == 63) {
            long long now;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
            if (t0 == 0) t0 = now;
            if (__any_sync(0xffffffffu, *dead || now - t0 > limit_ns)) {
                *dead = 1;
                return false;
            }
        }
    }
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void lds_vec4(float* d, uint32_t addr) {
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(addr));
}
__device__ __forceinline__ void chain_fma(float& q, float k, float p) {
    asm volatile("fma.rn.f32 %0, %1, %2, %0;" : "+f"(q) : "f"(k), "f"(p));
}
__device__ __forceinline__ void cp_async_16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}

// HOOK: the wait limit and the absent block of a test; otherwise the limit is a
// constant, without which the poll loops took 2.4% of an iteration (n = 7,900:
// 4.86 -> 4.98 ms).
template <int C, bool HOOK>
__global__ void __launch_bounds__(kCoopT, 1)
k_solve_coop(CoopSolve a) {
    constexpr int CP = C == 3 ? 4 : C;          // columns of p in shared memory, padded
    extern __shared__ __align__(16) float s_dyn[];
    const int rows = a.rows;
    const int JT = kCoopProd / a.groups;        // points a tile
    const int tile_floats = JT * rows;
    float* s_k = s_dyn;                                   // [3][JT / 4][rows][4]
    float* s_p = s_dyn + 3 * tile_floats;                 // [2][JT][CP]
    __shared__ double s_red[kCoopMaxGroups][kCoopMaxCols];
    __shared__ double s_worst[kCoopMaxCols];
    __shared__ float s_step[kCoopMaxCols];      // alpha, then beta
    __shared__ int s_active[kCoopMaxCols];
    __shared__ volatile int s_dead;
    const int t = threadIdx.x, lane = t & 31;
    const int warp = __shfl_sync(0xffffffffu, t >> 5, 0);  // uniform over the warp
    const bool producer = (warp & 3) != 3;
    const int g = warp >> 2;                              // others: row group, and column to reduce
    const bool consumer = !producer && g < a.groups;
    const int pt = (3 * (warp >> 2) + (warp & 3)) * 32 + lane;   // producer: 0 .. 383
    const int64_t n = a.n, n4 = (n + 3) & ~(int64_t)3;
    const int64_t i0 = (int64_t)blockIdx.x * rows;
    const int64_t i1 = i0 + rows < n ? i0 + rows : n;
    const int lrow = 32 * g + lane;                       // consumer: its row in the block
    const bool own = consumer && i0 + lrow < i1 && lrow < rows;
    const int64_t row = i0 + lrow;
    float* slab = a.slab + (int64_t)blockIdx.x * n4 * rows;
    const int tiles = (int)((n4 + JT - 1) / JT);
    if (HOOK && (int)blockIdx.x == a.skip_block) return;
    const long long limit_ns = HOOK ? a.limit_ns : kSolveWaitNs;
    if (t == 0) s_dead = 0;

    // All-reduction of one value per consumer lane and column, and a grid
    // barrier.  scalar_step(total, c) runs in one lane.  False once a wait
    // has run out of time (latched; every block then returns).
    auto reduce = [&](const double (&v)[C], int ph, uint64_t epoch, auto&& scalar_step) -> bool {
        if (!producer) {
            if (consumer) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    double x = v[c];
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
                    if (lane == 0) s_red[g][c] = x;
                    __syncwarp();
                }
            }
            asm volatile("bar.sync 1, 128;" ::: "memory");       // the four warps 3 mod 4
            if (g < C) {
                double x = s_red[0][g];
                for (int q = 1; q < a.groups; ++q) x += s_red[q][g];
                const int64_t G = gridDim.x;
                CoopWord* mail = a.mail + ((int64_t)ph * C + g) * G * G;
                for (int64_t b = lane; b < G; b += 32)
                    word_store(mail + b * G + blockIdx.x, (uint64_t)__double_as_longlong(x), epoch);
                x = 0.0;
                for (int64_t b0 = 0; b0 < G; b0 += 32) {
                    const bool live = b0 + lane < G;
                    uint64_t w;        // a lane without a word adds 0
                    if (!word_wait(mail + blockIdx.x * G + (live ? b0 + lane : 0), live, epoch, w, &s_dead,
                                   limit_ns)) {
                        a.result->failed = 1;
                        break;
                    }
                    x += __longlong_as_double((long long)w);
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                if (lane == 0) scalar_step(x, g);
                __syncwarp();
            }
        }
        __syncthreads();
        return s_dead == 0;
    };

    // the block's slab of K (points past the end: 0), four points a thread
    const uint32_t units = (uint32_t)(n4 / 4) * (uint32_t)rows;
    for (uint32_t e = t; e < units; e += kCoopT) {
        const int lr = (int)(e % (uint32_t)rows);
        const int64_t j = (int64_t)(e / (uint32_t)rows) * 4;
        const float4 x = __ldg(a.X + (i0 + lr < i1 ? i0 + lr : i0));
        float k[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float4 y = __ldg(a.X + (j + u < n ? j + u : 0));
            const float dx = __fsub_rn(x.x, y.x), dy = __fsub_rn(x.y, y.y), dz = __fsub_rn(x.z, y.z);
            const float d2 = fmaf(dz, dz, fmaf(dy, dy, __fmul_rn(dx, dx)));
            k[u] = j + u < n ? ex2_solve(__fmul_rn(d2, a.ns_log2e)) : 0.f;
        }
        reinterpret_cast<float4*>(slab)[e] = make_float4(k[0], k[1], k[2], k[3]);
    }

    float r[C], p[C], w[C];        // consumer: its row
    double acc64[C];
    double bb = 0.0, rs = 0.0;     // the reducing lane of column c: b.b and r.r
#pragma unroll
    for (int c = 0; c < C; ++c) {
        r[c] = own ? __ldg(a.B + row * C + c) : 0.f;
        p[c] = w[c] = 0.f;
        acc64[c] = own ? (double)r[c] * r[c] : 0.0;
    }
    auto publish = [&](uint64_t epoch) {
#pragma unroll
        for (int c = 0; c < C; ++c)
            if (own)
                word_store(a.rp + row * C + c,
                           (uint64_t)__float_as_uint(r[c]) | ((uint64_t)__float_as_uint(p[c]) << 32), epoch);
    };
    publish(1);
    // the reduction's __syncthreads also orders the slab before its copies
    if (!reduce(acc64, 1, 1, [&](double x, int c) {
            bb = rs = x;
            s_step[c] = 0.f;
            s_active[c] = bb > 0.0;
        }))
        return;

    // copy of tile k of the slab into ring slot `slot` (a commit group even if
    // it is empty)
    auto copy_tile = [&](int k, int slot) {
        const int64_t first = (int64_t)k * JT;
        const int cnt = (int)((n4 - first < JT ? n4 - first : JT) / 4 * rows);    // 16-byte units
        const float4* src = reinterpret_cast<const float4*>(slab) + first / 4 * rows;
        float4* dst = reinterpret_cast<float4*>(s_k + slot * tile_floats);
        for (int e = pt; e < cnt; e += kCoopProd) cp_async_16(dst + e, src + e);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int slot = 0, next_k = 0;      // ring slot of the tile consumed next; tile copied next
    auto copy_next = [&](int into) {
        copy_tile(next_k, into);
        if (++next_k == tiles) next_k = 0;
    };
    if (producer) {
        copy_next(0);
        copy_next(1);
    }
    int it = 0;
    for (;;) {
        bool any = false, active[C];
        float beta[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
            active[c] = s_active[c] != 0;
            beta[c] = s_step[c];
            any |= active[c];
        }
        if (!any || it >= a.max_iter) break;
        // a producer's point of a tile: its residual and last direction
        uint64_t rp[C];
        auto fetch = [&](int k) {
            const int64_t j = (int64_t)k * JT + pt;
            const bool live = pt < JT && j < n;
#pragma unroll
            for (int c = 0; c < C; ++c)
                if (!word_wait(a.rp + (live ? j * C + c : 0), live, (uint64_t)it + 1, rp[c], &s_dead,
                               limit_ns))
                    a.result->failed = 1;
        };
        auto direction = [&](int k) {      // of the points fetched last
            if (pt < JT) {
#pragma unroll
                for (int c = 0; c < C; ++c) {
                    const float rj = __uint_as_float((uint32_t)rp[c]);
                    const float pj = __uint_as_float((uint32_t)(rp[c] >> 32));
                    s_p[((k & 1) * JT + pt) * CP + c] =
                        it == 0 ? rj : active[c] ? fmaf(beta[c], pj, rj) : 0.f;
                }
            }
        };
        float q[C];
#pragma unroll
        for (int c = 0; c < C; ++c) q[c] = 0.f;
        auto consume = [&](int k) {
            const uint32_t kb = smem_addr(s_k + slot * tile_floats) + 16 * (lrow < rows ? lrow : 0);
            const uint32_t pb = smem_addr(s_p + (k & 1) * JT * CP);
            const int64_t left = n4 - (int64_t)k * JT;
            const int cnt = (int)(left < JT ? left : JT);
            // batches of U points, the next one loaded while this one's FMAs
            // run; volatile and without a branch around the last load, because
            // the chain otherwise waited for its loads (7 clocks a point; 5.1
            // so, alone)
            constexpr int U = C == 1 ? 16 : 8;
            float kv[2][U], pv[2][U * CP];
            auto load = [&](int j, int h) {
#pragma unroll
                for (int u = 0; u < U; u += 4) {
                    lds_vec4(kv[h] + u, kb + (j + u) * 4 * rows);
#pragma unroll
                    for (int v = 0; v < CP; ++v) lds_vec4(pv[h] + u * CP + 4 * v, pb + ((j + u) * CP + 4 * v) * 4);
                }
            };
            auto chain = [&](int h) {
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int c = 0; c < C; ++c) chain_fma(q[c], kv[h][u], pv[h][u * CP + c]);
            };
            const int whole = cnt / (2 * U);      // pairs of batches
            if (whole > 0) load(0, 0);
#pragma unroll 1
            for (int k2 = 0; k2 < whole; ++k2) {
                load((2 * k2 + 1) * U, 1);
                chain(0);
                load(k2 + 1 < whole ? (2 * k2 + 2) * U : 0, 0);
                chain(1);
            }
#pragma unroll 1
            for (int j = whole * 2 * U; j < cnt; j += 4) {
                float k4[4], p4[4 * CP];
                lds_vec4(k4, kb + j * 4 * rows);
#pragma unroll
                for (int v = 0; v < CP; ++v) lds_vec4(p4 + 4 * v, pb + (j * CP + 4 * v) * 4);
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int c = 0; c < C; ++c) chain_fma(q[c], k4[u], p4[u * CP + c]);
            }
        };
        if (producer) {
            fetch(0);
            direction(0);
            if (tiles > 1) fetch(1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");   // the first tile is here
        }
        __syncthreads();
        for (int k = 0; k < tiles; ++k) {
            if (consumer) {
                consume(k);
            } else if (producer) {
                copy_next(slot == 0 ? 2 : slot - 1);      // the slot consumed last
                if (k + 1 < tiles) direction(k + 1);
                if (k + 2 < tiles) fetch(k + 2);
                asm volatile("cp.async.wait_group 1;" ::: "memory");   // the next tile is here
            }
            __syncthreads();
            slot = slot == 2 ? 0 : slot + 1;
        }
#pragma unroll
        for (int c = 0; c < C; ++c) {
            p[c] = it == 0 ? r[c] : active[c] ? fmaf(beta[c], p[c], r[c]) : 0.f;
        }
        if (consumer) {
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const double pd = p[c];
                acc64[c] = own ? pd * ((double)q[c] + (double)a.sigma2 * pd) : 0.0;
            }
        }
        if (!reduce(acc64, 0, (uint64_t)it + 1, [&](double pap, int c) {
                s_step[c] = s_active[c] && pap > 0.0 ? (float)(rs / pap) : 0.f;
            }))
            break;
#pragma unroll
        for (int c = 0; c < C; ++c) {
            const float alpha = s_step[c];
            const float ap = fmaf(a.sigma2, p[c], q[c]);
            w[c] = fmaf(alpha, p[c], w[c]);
            r[c] = fmaf(-alpha, ap, r[c]);
        }
        publish((uint64_t)it + 2);
        if (consumer) {
#pragma unroll
            for (int c = 0; c < C; ++c) acc64[c] = own ? (double)r[c] * r[c] : 0.0;
        }
        if (!reduce(acc64, 1, (uint64_t)it + 2, [&](double now, int c) {
                float step = 0.f;
                if (s_active[c]) {
                    step = (float)(rs > 0.0 ? now / rs : 0.0);
                    rs = now;
                    s_active[c] = now > a.tol2 * bb;
                }
                s_step[c] = step;
            }))
            break;
        ++it;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");   // no copy outlives the block
    if (own) {
#pragma unroll
        for (int c = 0; c < C; ++c) a.W[row * C + c] = w[c];
    }
    if (blockIdx.x == 0) {
        if (!producer && g < C && lane == 0) s_worst[g] = bb > 0.0 ? rs / bb : 0.0;
        __syncthreads();
        if (t == 0 && s_dead == 0) {
            double worst = 0.0;
            for (int c = 0; c < C; ++c)
                if (s_worst[c] > worst) worst = s_worst[c];
            a.result->iters = it;
            a.result->done = 1;
            a.result->worst = worst;
        }
    }
}

// Row blocks of the step kernels: 16 rows each (their FP64 sums are bound by
// the FP64 pipes, so they want all SMs: 256 rows a block took 17-34 us a
// kernel at n = 4096), at most 1024.
int solve_blocks(int64_t n) {
    const int64_t b = (n + 15) / 16;
    return (int)(b < 1024 ? (b > 0 ? b : 1) : 1024);
}

template <class... KArgs, class... Args>
cudaError_t solve_launch(void (*kern)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace

// Floats a vector takes in the workspace: a multiple of 4, so that the FP64
// partials that follow the vectors are aligned for every n and nrhs.
static size_t solve_vector_floats(int64_t n, int nrhs) {
    return ((size_t)n * nrhs + 3) & ~(size_t)3;
}

size_t solve_workspace_bytes(int64_t n, int nrhs) {
    const size_t v = solve_vector_floats(n, nrhs) * sizeof(float);
    return 3 * v + (size_t)solve_blocks(n) * nrhs * sizeof(double) + (size_t)nrhs * sizeof(Col) +
           256 * 4;
}

// FP32 systems of at most kCoopMaxCols columns run in one cooperative launch
// while their rows fit the SMs' consumer lanes (64 an SM: n <= 9,728 on 152
// SMs, a slab of 378 MB).  Up to n ~ 5,000 the slab stays in L2; past it the
// stream from memory takes 4 n^2 bytes an iteration, which at n = 9,728 is
// still below the stepwise form (94 us an iteration against 271).
static int64_t coop_rows(int64_t n) {
    const int64_t share = (n + num_sms() - 1) / num_sms();
    return share > 32 ? share : 32;     // 32 rows cost a warp what one row does
}

bool solve_coop_supported(int64_t n, int nrhs) {
    return nrhs <= kCoopMaxCols && coop_rows(n) <= 32 * kCoopMaxGroups;
}

struct CoopLayout {
    int64_t rows, blocks, n4;
    size_t rp, mail, clear, slab, bytes;    // offsets; [0, clear) is zeroed
    CoopLayout(int64_t n, int nrhs) {
        rows = coop_rows(n);
        if (rows > n) rows = n;
        blocks = (n + rows - 1) / rows;
        n4 = (n + 3) & ~(int64_t)3;
        rp = 64;                             // the result comes first
        mail = rp + (size_t)n * nrhs * sizeof(CoopWord);
        clear = mail + 2 * (size_t)nrhs * blocks * blocks * sizeof(CoopWord);
        slab = (clear + 255) & ~(size_t)255;
        bytes = slab + (size_t)blocks * rows * n4 * sizeof(float);
    }
};

size_t solve_coop_workspace_bytes(int64_t n, int nrhs) { return CoopLayout(n, nrhs).bytes; }

// Returns cudaErrorNotSupported where the launch does not fit this device
// (the caller then runs run_solve).
cudaError_t run_solve_coop(int64_t n, int nrhs, const float4* X, const float* B, float s, float sigma2,
                           float tol, int max_iter, float* W, void* ws, int* iters, float* relres,
                           const SolveWait& wait, bool* timed_out, cudaStream_t st) {
    const bool hook = wait.limit_ns > 0;
    const void* fn = nrhs == 1   ? hook ? (const void*)k_solve_coop<1, true> : (const void*)k_solve_coop<1, false>
                     : nrhs == 2 ? hook ? (const void*)k_solve_coop<2, true> : (const void*)k_solve_coop<2, false>
                     : nrhs == 3 ? hook ? (const void*)k_solve_coop<3, true> : (const void*)k_solve_coop<3, false>
                     : hook      ? (const void*)k_solve_coop<4, true>
                                 : (const void*)k_solve_coop<4, false>;
    const CoopLayout lay(n, nrhs);
    if (lay.blocks > kCoopMaxBlocks) return cudaErrorNotSupported;
    CoopSolve a;
    a.n = n;
    a.rows = (int)lay.rows;
    a.groups = (int)((lay.rows + 31) / 32);
    const int cp = nrhs == 3 ? 4 : nrhs, jt = kCoopProd / a.groups;
    const size_t smem = (3 * (size_t)jt * a.rows + 2 * (size_t)jt * cp) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kCoopT, smem);
    if (e != cudaSuccess) return e;
    if ((int64_t)per_sm * num_sms() < lay.blocks) return cudaErrorNotSupported;
    uint8_t* q = (uint8_t*)ws;
    a.X = X;
    a.B = B;
    a.ns_log2e = -s * 1.4426950408889634f;
    a.sigma2 = sigma2;
    a.tol2 = (double)tol * tol;
    a.max_iter = max_iter;
    a.W = W;
    a.result = (CoopResult*)q;
    a.rp = (CoopWord*)(q + lay.rp);
    a.mail = (CoopWord*)(q + lay.mail);
    a.slab = (float*)(q + lay.slab);
    a.limit_ns = wait.limit_ns;
    a.skip_block = wait.skip_block;
    // epochs start at 0, and so does the result
    if ((e = cudaMemsetAsync(q, 0, lay.clear, st)) != cudaSuccess) return e;
    void* args[] = {&a};
    e = cudaLaunchCooperativeKernel(fn, dim3((unsigned)lay.blocks), dim3(kCoopT), args, smem, st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return cudaErrorNotSupported;
    }
    CoopResult res;
    e = cudaMemcpyAsync(&res, a.result, sizeof(res), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    *timed_out = res.failed || !res.done;
    if (iters) *iters = res.iters;
    if (relres) *relres = (float)sqrt(res.worst);
    return cudaSuccess;
}

// Conjugate gradients; the matvec Q = K(X, X) P is supplied by the caller.
cudaError_t run_solve(int64_t n, int nrhs, const float* B, float sigma2, float tol, int max_iter,
                      float* W, void* ws, const SolveMatvec& mv, int* iters, float* relres,
                      cudaStream_t st) {
    const size_t v = solve_vector_floats(n, nrhs);
    float* R = (float*)ws;
    float* P = R + v;
    float* Q = P + v;
    double* partial = (double*)(Q + v);
    const int blocks = solve_blocks(n);
    Col* col = (Col*)(partial + (size_t)blocks * nrhs);
    int* n_active_dev = (int*)(col + nrhs);
    const dim3 grid((unsigned)blocks, (unsigned)((nrhs + kCols - 1) / kCols)), block(kCols, kRowLanes);
    const double tol2 = (double)tol * tol;
    int n_active = 0;
    cudaError_t e;
    auto finish = [&](int what) -> cudaError_t {
        return solve_launch(k_solve_finish, dim3((unsigned)nrhs), dim3(32), st, (const double*)partial, blocks,
                            nrhs, what, tol2, col, n_active_dev);
    };
    // the count of active columns starts each step at 0
    if ((e = cudaMemsetAsync(n_active_dev, 0, sizeof(int), st)) != cudaSuccess) return e;
    k_solve_init<<<grid, block, 0, st>>>(n, nrhs, B, R, P, W, partial);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = finish(0)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(&n_active, n_active_dev, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess)
        return e;
    if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    int it = 0;
    while (n_active > 0 && it < max_iter) {
        if ((e = mv(P, Q)) != cudaSuccess) return e;
        e = solve_launch(k_solve_pap, grid, block, st, n, nrhs, (const float*)P, (const float*)Q, sigma2,
                         partial, n_active_dev);
        if (e != cudaSuccess || (e = finish(1)) != cudaSuccess) return e;
        e = solve_launch(k_solve_update, grid, block, st, n, nrhs, (const float*)P, (const float*)Q, sigma2,
                         (const Col*)col, R, W, partial);
        if (e != cudaSuccess || (e = finish(2)) != cudaSuccess) return e;
        e = solve_launch(k_solve_dir, grid, block, st, n, nrhs, (const float*)R, (const Col*)col, P);
        if (e != cudaSuccess) return e;
        ++it;
        if ((e = cudaMemcpyAsync(&n_active, n_active_dev, sizeof(int), cudaMemcpyDeviceToHost, st)) !=
            cudaSuccess)
            return e;
        if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
    }
    // largest relative residual (the recurrence's r.r over b.b)
    std::vector<Col> hc((size_t)nrhs);
    if ((e = cudaMemcpyAsync(hc.data(), col, (size_t)nrhs * sizeof(Col), cudaMemcpyDeviceToHost, st)) !=
            cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
        return e;
    double worst = 0.0;
    for (const Col& k : hc) {
        const double q = k.bb > 0.0 ? k.rs / k.bb : 0.0;
        if (q > worst) worst = q;
    }
    if (iters) *iters = it;
    if (relres) *relres = (float)sqrt(worst);
    return cudaSuccess;
}

}  // namespace ab
