// Step a2: pivoted Cholesky of a positive semidefinite Hankel block, O(K^2 N), in float64
// (Sec. 2.1, Fig. 2).
//
// Only the diagonal d and the K selected columns are ever formed.  Step r:
//   p_r = argmax_j d_j                      (lowest index on ties)
//   c   = H[:, p_r] - sum_{i<r} u_i u_i[p_r]   (earlier steps applied to column p_r)
//   a_r = c[p_r];  u_r = c / sqrt(a_r);  d <- d - u_r^2
// and the factorisation stops before any step whose pivot (max d, or a_r) is
// <= tol * max(diag H).  u_r = l_r / sqrt(a_r) in the paper's notation, so
// H ~ sum_r l_r l_r^T / a_r = sum_r u_r u_r^T.
//
// One launch for all steps: a block owns a fixed slice of indices, publishes the argmax of its slice
// of the updated d, and after a grid-wide barrier every block reduces the few hundred entries to the
// pivot and takes the same stop decision from the same data.  The blocks fit the device all at once,
// but beside other work, or where the process may not use every SM, they need not be resident
// together, so nothing relies on it: the barrier's waits are bounded, a wait that runs out ends the
// launch, and the factorisation then runs as one launch per step, whose blocks wait for nobody.
// Latency-bound, a step is one chain of dependent loads: plan creation at n = 2^16 takes 650 us in
// one launch, 720 us in one per step.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "tdh_internal.cuh"

namespace tdh {
namespace {

constexpr int kThreads = 256;
constexpr int kKmaxShared = kPcholSteps;  // u_i[p] for i < r staged in shared memory

struct State {
    double thresh;  // tol * max(diag H)
    int64_t K;      // steps taken
    int done;
    int timeout;    // a barrier's wait ran out
    unsigned count; // the barrier
};

// What a block publishes of its slice after a step: the largest residual diagonal entry (its
// value as an ordered integer, the lowest index on ties) and, for accuracy-targeted runs, the
// factors of the truncation bound as bit patterns.  All comparisons are integer ones: a float64
// comparison takes the SM's two float64 lanes sixteen cycles a warp, and the reductions need
// hundreds of them.
struct __align__(16) Part {
    int64_t key;
    int64_t i;
    int64_t b1, b2;  // max (D1_j / w_j)^2 d_j, max (D2_j / w_j)^2 d_j (not below 0)
};

// Accuracy target of a run (a1 null: none): a1_j = (D1_j / w_j)^2, a2_j = (D2_j / w_j)^2 (with
// the step's scalings), tmax = max |t|.
struct TargetSpec {
    const double* a1;
    const double* a2;
    const double* tmax;
    double target;
};

// Doubles in the order of signed integers (NaN below everything), and back.
__device__ __forceinline__ int64_t order_key(double v) {
    const int64_t b = __double_as_longlong(v);
    return v == v ? b ^ ((b >> 63) & INT64_MAX) : INT64_MIN;
}
__device__ __forceinline__ double order_value(int64_t k) {
    return __longlong_as_double(k ^ ((k >> 63) & INT64_MAX));
}

__device__ __forceinline__ Part pmax(Part a, Part b) {
    const bool second = b.key > a.key || (b.key == a.key && b.i < a.i);
    Part r;
    r.key = second ? b.key : a.key;
    r.i = second ? b.i : a.i;
    r.b1 = b.b1 > a.b1 ? b.b1 : a.b1;
    r.b2 = b.b2 > a.b2 ? b.b2 : a.b2;
    return r;
}

__device__ __forceinline__ Part part_none() { return Part{INT64_MIN, INT64_MAX, 0, 0}; }

__device__ __forceinline__ Part warp_max(Part x) {
    for (int off = 16; off > 0; off >>= 1) {
        Part o;
        o.key = __shfl_xor_sync(0xffffffffu, x.key, off);
        o.i = __shfl_xor_sync(0xffffffffu, x.i, off);
        o.b1 = __shfl_xor_sync(0xffffffffu, x.b1, off);
        o.b2 = __shfl_xor_sync(0xffffffffu, x.b2, off);
        x = pmax(x, o);
    }
    return x;
}

// Entry j's share of the block's maxima, residual diagonal dj (j >= j0).
__device__ __forceinline__ Part part_of(const TargetSpec& T, int64_t j, double dj, bool in) {
    Part p{order_key(dj), j, 0, 0};
    if (T.a1 && in && dj > 0.0) {  // (a negative rounding residue counts as 0)
        p.b1 = __double_as_longlong(T.a1[j] * dj);
        p.b2 = __double_as_longlong(T.a2[j] * dj);
    }
    return p;
}

__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// The maximum of the block's values to part[blockIdx.x].
__device__ __forceinline__ void publish(Part own, Part* s_part, Part* part) {
    own = warp_max(own);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = own;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < kThreads / 32; ++i) own = pmax(own, s_part[i]);
        part[blockIdx.x] = own;
    }
}

// Grid-wide barrier, for the gen-th time: blocks count up to gen gridDim.x (+ stall, for a test of
// the limit).  Returns false when the wait, or another block's, ran out.
constexpr long long kBarrierNs = 100000000ll;
__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ bool grid_barrier(State* st, unsigned gen, unsigned stall) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&st->count, 1u);
        const unsigned goal = gen * gridDim.x + stall;
        const long long t0 = global_ns();
        int good = 1;
        while (*(volatile unsigned*)&st->count < goal) {
            if (*(volatile int*)&st->timeout || global_ns() - t0 > kBarrierNs) {
                good = 0;
                break;
            }
        }
        __threadfence();
        ok = good;
    }
    __syncthreads();
    return ok != 0;
}

// d_j = H_jj = h[2j] of the block's slice for j >= j0 (excluded indices get -inf); their maximum
// goes to part[blockIdx.x].
__device__ __forceinline__ void init_slice(const double* h, int64_t n, int64_t j0, const double* w,
                                           const TargetSpec& T, double* d, Part* part,
                                           Part* s_part) {
    Part own = part_none();
    for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < n;
         j += (int64_t)gridDim.x * kThreads) {
        const double v = (j >= j0) ? h[2 * j] * (w ? w[j] * w[j] : 1.0) : -INFINITY;
        d[j] = v;
        own = pmax(own, part_of(T, j, v, j >= j0));
    }
    publish(own, s_part, part);
}

__global__ void __launch_bounds__(kThreads) pchol_init(const double* __restrict__ h, int64_t n,
                                                       int64_t j0, const double* __restrict__ w,
                                                       TargetSpec T, double* d, Part* part) {
    __shared__ Part s_part[kThreads / 32];
    pdl_trigger();
    init_slice(h, n, j0, w, T, d, part, s_part);
}

// ALL: every step (r0 = 0); else step r0, overlapping the end of the kernel before it.  Warp 0
// decides, gathers the pivot row of the factors and forms its scale; the column's dot products
// read the earlier factors kBatch at a time (independent loads in flight), and subtract in order.
// What other blocks wrote is read past L1.  part: [2][gridDim.x], alternating between steps.
constexpr int kBatch = 8;

template <bool ALL>
__global__ void __launch_bounds__(kThreads, 2) pchol_step(
    const double* __restrict__ h, int64_t n, int64_t j0, const double* __restrict__ w, double tol,
    TargetSpec T, int r0, int kmax, double* u, int64_t* __restrict__ piv, double* d, Part* part,
    State* st, unsigned stall) {
    __shared__ double s_up[kKmaxShared];
    __shared__ Part s_part[kThreads / 32];
    __shared__ double s_inv, s_wp;
    __shared__ int64_t s_p;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool lead = blockIdx.x == 0 && threadIdx.x == 0;
    const double tmax = T.a1 ? *T.tmax : 0.0;
    const int64_t jf = (int64_t)blockIdx.x * kThreads + threadIdx.x;  // this thread's first index
    if constexpr (ALL) {
        init_slice(h, n, j0, w, T, d, part, s_part);
    } else {
        pdl_trigger();
        pdl_wait();
    }
    for (int r = r0; ALL ? r < kmax : r == r0; ++r) {
        if (ALL && !grid_barrier(st, (unsigned)r + 1u, stall)) {
            if (threadIdx.x == 0) st->timeout = 1;
            return;
        }
        // every block reduces the same partials: identical pivot and decision everywhere
        const Part* in = part + (r & 1) * (int)gridDim.x;
        Part best = part_none();
        for (int i = threadIdx.x; i < gridDim.x; i += kThreads) {
            const longlong2* q = reinterpret_cast<const longlong2*>(in + i);
            const longlong2 a = __ldcg(q), b = __ldcg(q + 1);
            best = pmax(best, Part{a.x, a.y, b.x, b.y});
        }
        best = warp_max(best);
        if (lane == 0) s_part[warp] = best;
        __syncthreads();
        if (warp == 0) {
            best = warp_max(lane < kThreads / 32 ? s_part[lane] : part_none());
            const int64_t p = best.i;
            // One thread reads the state: block 0 may set `done` while other blocks of this step
            // still look at it, so the threads of a block must not each decide from their own
            // reading.  (A block that sees this step's `done` stops as its own data would have it.)
            int stop = 0, done = 0;
            double thresh = 0.0;
            if (lane == 0) {
                const double v = order_value(best.key);
                if (!ALL) done = *(volatile int*)&st->done;
                thresh = r == 0 ? tol * v : *(volatile double*)&st->thresh;
                const bool met = T.a1 && tmax * sqrt(__longlong_as_double(best.b1)) *
                                                 sqrt(__longlong_as_double(best.b2)) <= T.target;
                stop = done || met || !(v > thresh) || p < j0 || p >= n;
            }
            stop = __shfl_sync(0xffffffffu, stop, 0);
            if (!stop) {
                const double wp = w ? w[p] : 1.0, hp = h[2 * p];
                for (int i = lane; i < r; i += 32) s_up[i] = __ldcg(u + (int64_t)i * n + p);
                __syncwarp();
                if (lane == 0) {
                    double a = hp * wp * wp;
                    for (int i = 0; i < r; ++i) a -= s_up[i] * s_up[i];
                    if (!(a > thresh)) stop = 1;
                    s_wp = wp;
                    s_inv = 1.0 / sqrt(a);
                }
            }
            if (lane == 0) s_p = stop ? -1 : p;
            if (lead && !done) {  // (only this thread ever sets `done`)
                st->K = stop ? r : r + 1;
                if (stop) st->done = 1;
                if (r == 0) st->thresh = thresh;
            }
        }
        __syncthreads();
        const int64_t p = s_p;
        if (p < 0) return;
        const double wp = s_wp;
        const double inv = s_inv;
        Part own = part_none();
        double* ur = u + (int64_t)r * n;
        for (int64_t j = jf; j < n; j += (int64_t)gridDim.x * kThreads) {
            double val = 0.0;
            double dj = -INFINITY;
            if (j >= j0) {
                double c = h[j + p] * (w ? w[j] * wp : 1.0);
                const double dold = __ldcg(d + j);
                const double* uj = u + j;
                int i = 0;
                for (; i + kBatch <= r; i += kBatch) {
                    double x[kBatch];
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) x[b] = __ldcg(uj + (int64_t)(i + b) * n);
#pragma unroll
                    for (int b = 0; b < kBatch; ++b) c -= x[b] * s_up[i + b];
                }
                for (; i < r; ++i) c -= __ldcg(uj + (int64_t)i * n) * s_up[i];
                val = c * inv;
                dj = dold - val * val;
                d[j] = dj;
            }
            ur[j] = val;
            own = pmax(own, part_of(T, j, dj, j >= j0));
        }
        publish(own, s_part, part + ((r + 1) & 1) * (int)gridDim.x);
        if (lead) piv[r] = p;
    }
}

}  // namespace

namespace {

// The steps of a factorisation on stream s: state, residual diagonal and partials given (2 nblk of
// them).  Launch by launch, the host reads the stop state after kFirstSteps, then every kNextSteps
// steps; those launched past the end return at once.
constexpr int64_t kFirstSteps = 20, kNextSteps = 12;

cudaError_t read_state(State* host, const State* st, cudaStream_t s) {
    cudaError_t e = cudaMemcpyAsync(host, st, sizeof(State), cudaMemcpyDeviceToHost, s);
    return e == cudaSuccess ? cudaStreamSynchronize(s) : e;
}

cudaError_t pchol_steps(const double* h, const double* w, int64_t n, int64_t j0, double tol,
                        int64_t kmax, const TargetSpec& T, double* u, int64_t* pivots, double* d,
                        Part* part, int nblk, State* st, State* host, cudaStream_t s) {
    *host = State{};
    cudaError_t e = cudaMemsetAsync(st, 0, sizeof(State), s);
    if (e == cudaSuccess) {
        pchol_step<true><<<nblk, kThreads, 0, s>>>(h, n, j0, w, tol, T, 0, (int)kmax, u, pivots, d,
                                                   part, st, tc_stall_enabled() ? 1u : 0u);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = read_state(host, st, s);
    if (e != cudaSuccess || !host->timeout) return e;
    // not all of its blocks were resident: from the start again, a launch per step
    e = cudaMemsetAsync(st, 0, sizeof(State), s);
    if (e == cudaSuccess) {
        pchol_init<<<nblk, kThreads, 0, s>>>(h, n, j0, w, T, d, part);
        e = cudaGetLastError();
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)nblk);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int64_t poll = kFirstSteps;
    for (int64_t r = 0; e == cudaSuccess && r < kmax; ++r) {
        e = cudaLaunchKernelEx(&cfg, pchol_step<false>, h, n, j0, w, tol, T, (int)r, (int)kmax, u,
                               pivots, d, part, st, 0u);
        if (e == cudaSuccess && (r + 1 == poll || r + 1 == kmax)) {
            poll += kNextSteps;
            e = read_state(host, st, s);
            if (host->done) break;
        }
    }
    return e;
}

}  // namespace

// Blocks of the launch: all resident at once on an idle device (two of at most 128 registers a
// thread per SM).
int pchol_blocks(int64_t n) {
    return (int)std::max<int64_t>(
        1, std::min<int64_t>((n + kThreads - 1) / kThreads, 2 * (int64_t)sm_count()));
}

int pchol_run(const double* h, const double* w, int64_t n, int64_t j0, double tol, int64_t kmax,
              const PcholTarget* target, double* u, int64_t* pivots, int64_t* K, cudaStream_t s) {
    if (kmax > kKmaxShared) kmax = kKmaxShared;
    if (kmax > n - j0) kmax = n - j0;
    const int nblk = pchol_blocks(n);
    double* d = nullptr;
    Part* part = nullptr;
    State* st = nullptr;
    int rc = TDH_OK;
    State host{};
    TargetSpec T{};
    if (target) T = TargetSpec{target->a1, target->a2, target->tmax, target->tol};
    if ((rc = dev_alloc_t(&d, (size_t)n)) != TDH_OK) goto done;
    if ((rc = dev_alloc_t(&part, (size_t)2 * nblk)) != TDH_OK) goto done;
    if ((rc = dev_alloc_t(&st, 1)) != TDH_OK) goto done;
    {
        const cudaError_t e =
            pchol_steps(h, w, n, j0, tol, kmax, T, u, pivots, d, part, nblk, st, &host, s);
        if (e != cudaSuccess) {
            set_error("pivoted Cholesky: %s", cudaGetErrorString(e));
            rc = TDH_ERR_CUDA;
        }
    }
    if (rc == TDH_OK) *K = host.K;
done:
    if (d || part || st) cudaStreamSynchronize(s);
    dev_free(d);
    dev_free(part);
    dev_free(st);
    return rc;
}

// ----------------------------------------------------------------------------------------
// Accuracy-targeted truncation.  The residual R = H - sum_{r<K} u_r u_r^T of a pivoted
// Cholesky of a positive semidefinite H is positive semidefinite (a Schur complement), so each
// 2 x 2 principal minor gives |R_jk| <= sqrt(d_j d_k) with d = diag(R).  In A = D1 (T o H) D2
// the truncation error is then |(A - A_K)_jk| <= max|t| |D1_j| sqrt(d_j) |D2_k| sqrt(d_k), and
// max |beta_K - beta| <= B(K) ||alpha||_1 with B(K) = max|t| max_j |D1_j| sqrt(d_j)
// max_k |D2_k| sqrt(d_k).  A run with a target stops at the first K whose B(K) meets it: every
// step publishes B's two maxima beside the next pivot, so the steps beyond K, up to the rounding
// floor, are never taken (128 steps and 3.7 ms at n = 1024 where 11 are kept).
namespace {

// w_j = sqrt(|D1_j D2_j|) (with the step's scalings), 1 where that is 0 or not finite; a1_j =
// (D1_j / w_j)^2, a2_j = (D2_j / w_j)^2 (0 for j < j0); *tmax = max |t_j| (cleared before the
// launch; non-negative doubles order like their bit patterns).
__global__ void __launch_bounds__(kThreads) k_pivot_weights(
    const double* __restrict__ t, const double* __restrict__ d1, const double* __restrict__ d2,
    const double* __restrict__ so, const double* __restrict__ si, int64_t n, int64_t j0,
    double* __restrict__ w, double* __restrict__ a1, double* __restrict__ a2,
    unsigned long long* __restrict__ tmax) {
    const int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    double tm = 0.0;
    if (j < n) {
        const double x1 = fabs(d1[j] * (so ? so[j] : 1.0)), x2 = fabs(d2[j] * (si ? si[j] : 1.0));
        const double v = sqrt(fabs(d1[j] * (so ? so[j] : 1.0) * d2[j] * (si ? si[j] : 1.0)));
        const double wj = (v > 0.0 && isfinite(v)) ? v : 1.0;
        w[j] = wj;
        const double r1 = x1 / wj, r2 = x2 / wj;
        a1[j] = j >= j0 ? r1 * r1 : 0.0;
        a2[j] = j >= j0 ? r2 * r2 : 0.0;
        tm = fabs(t[j]);
    }
    for (int off = 16; off > 0; off >>= 1) tm = fmax(tm, __shfl_xor_sync(0xffffffffu, tm, off));
    if ((threadIdx.x & 31) == 0) atomicMax(tmax, (unsigned long long)__double_as_longlong(tm));
}

// u[r][j] /= w_j: factors of W H W -> factors of H
__global__ void k_unweight(double* __restrict__ u, const double* __restrict__ w, int64_t K,
                           int64_t n) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < K * n) u[i] /= w[i % n];
}

}  // namespace

int pchol_weights(const double* t, const double* d1, const double* d2, const double* so,
                  const double* si, int64_t n, int64_t j0, double* w, double* a1, double* a2,
                  double* tmax, cudaStream_t s) {
    TDH_CUDA(cudaMemsetAsync(tmax, 0, sizeof(double), s));
    k_pivot_weights<<<(unsigned)((n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
        t, d1, d2, so, si, n, j0, w, a1, a2, reinterpret_cast<unsigned long long*>(tmax));
    TDH_CUDA(cudaGetLastError());
    return TDH_OK;
}

int pchol_unweight(double* u, const double* w, int64_t K, int64_t n, cudaStream_t s) {
    if (K <= 0) return TDH_OK;
    k_unweight<<<(unsigned)((K * n + kThreads - 1) / kThreads), kThreads, 0, s>>>(u, w, K, n);
    TDH_CUDA(cudaGetLastError());
    return TDH_OK;
}

}  // namespace tdh

extern "C" int tdh_pchol(const double* h, int64_t n, int64_t j0, double tol, int64_t kmax,
                         double* u, int64_t* pivots, int64_t* K, void* stream) {
    tdh::clear_error();
    if (n < 1 || (j0 != 0 && j0 != 1) || j0 >= n || !(tol > 0.0) || kmax < 1 || !h || !u ||
        !pivots || !K) {
        tdh::set_error("tdh_pchol: need n >= 1, j0 in {0,1} < n, tol > 0, kmax >= 1, non-NULL");
        return TDH_ERR_INVALID_ARG;
    }
    return tdh::pchol_run(h, nullptr, n, j0, tol, kmax, nullptr, u, pivots, K,
                          tdh::as_stream(stream));
}

// ----------------------------------------------------------------------------------------
// Allocation-free pivoted Cholesky.
//
// Some callers cannot call cudaMalloc at all: code that runs while a caching allocator owns
// the device memory and forbids outside allocations, or inside allocation-free real-time
// sections.  This variant runs the same kernels as tdh_pchol but takes its scratch (the
// residual diagonal, the per-block argmax partials and the stop state) from one statically
// sized device array that lives in this file.  The array is part of the library image: every
// GPU that loads the library holds it until the process exits.
//
// Every call looks up the array's device address for the current device with
// cudaGetSymbolAddress (a lookup, not an allocation) and passes it to the kernels, so the
// address is always the one of the current context.  All calls on a device share the one
// array and it keeps the contents of the last call: the state words that must start at zero
// are cleared by every call, the rest is fully rewritten.  Two calls whose work overlaps on
// the GPU (different streams, or different host threads) race on the array; serialise them.
// Each call synchronises `stream` (it reads the stop state back).
namespace tdh {
namespace {

constexpr int64_t kNoAllocMaxN = 65536;
constexpr int kNoAllocMaxParts = (int)((kNoAllocMaxN + kThreads - 1) / kThreads);
constexpr size_t kNoAllocDBytes = sizeof(double) * (size_t)kNoAllocMaxN;
constexpr size_t kNoAllocPartBytes = sizeof(Part) * 2 * (size_t)kNoAllocMaxParts;
constexpr size_t kNoAllocBytes = kNoAllocDBytes + kNoAllocPartBytes + 256;

static __device__ __align__(256) unsigned char g_pchol_scratch[kNoAllocBytes];

int noalloc_scratch(unsigned char** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_pchol_scratch);
    if (e != cudaSuccess || !p) {
        set_error("tdh_pchol_noalloc: cudaGetSymbolAddress failed: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    *out = static_cast<unsigned char*>(p);
    return TDH_OK;
}

}  // namespace
}  // namespace tdh

extern "C" int tdh_pchol_noalloc(const double* h, int64_t n, int64_t j0, double tol,
                                 int64_t kmax, double* u, int64_t* pivots, int64_t* K,
                                 void* stream) {
    using namespace tdh;
    clear_error();
    if (n < 1 || (j0 != 0 && j0 != 1) || j0 >= n || !(tol > 0.0) || kmax < 1 || !h || !u ||
        !pivots || !K) {
        set_error("tdh_pchol_noalloc: need n >= 1, j0 in {0,1} < n, tol > 0, kmax >= 1, non-NULL");
        return TDH_ERR_INVALID_ARG;
    }
    if (n > kNoAllocMaxN) {
        set_error("tdh_pchol_noalloc: n = %lld exceeds the static scratch limit of %lld "
                  "coefficients; use tdh_pchol", (long long)n, (long long)kNoAllocMaxN);
        return TDH_ERR_INVALID_ARG;
    }
    unsigned char* base = nullptr;
    TDH_TRY(noalloc_scratch(&base));
    cudaStream_t s = as_stream(stream);
    double* d = reinterpret_cast<double*>(base);
    Part* part = reinterpret_cast<Part*>(base + kNoAllocDBytes);
    State* st = reinterpret_cast<State*>(base + kNoAllocDBytes + kNoAllocPartBytes);
    if (kmax > kKmaxShared) kmax = kKmaxShared;
    if (kmax > n - j0) kmax = n - j0;
    // the same grid as tdh_pchol, within the array's partials
    const int nblk = pchol_blocks(n);
    State host{};
    const cudaError_t e = pchol_steps(h, nullptr, n, j0, tol, kmax, TargetSpec{}, u, pivots, d, part,
                                      nblk, st, &host, s);
    if (e != cudaSuccess) {
        set_error("tdh_pchol_noalloc: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    *K = host.K;
    return TDH_OK;
}
