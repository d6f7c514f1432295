// Case 1 of the ultraspherical (Sec. 5.2) and Jacobi (Sec. 5.3) conversions: when the two
// parameters differ by an integer, A is a product of sparse upper-triangular factors, each
// applied in O(n) (Eq. (12) and its Jacobi analogue).  A factor is
//   (S c)_j = p_j c_j + q_j c_{j+off}
// with
//   ultraspherical S_l (C^(l) -> C^(l+1)), off = 2:  p_j = l/(l+j),  q_j = -l/(l+j+2);
//   Jacobi S_(a,b) ((a,b) -> (a+1,b)), off = 1:
//       p_0 = 1,  p_j = (j+a+b+1)/(2j+a+b+1),  q_j = -(j+b+1)/(2j+a+b+3)
// (the superdiagonal numerator is j+b+1: that is what the exact conversion gives; the form
// with j+a+1 is the factor for raising b, up to sign).  Inside a reflected part of a Jacobi
// chain each factor is conjugated by diag((-1)^k), which negates q.  A step to a smaller
// parameter applies the inverses: S x = c is solved by back-substitution (Sec. 5.2, 5.3:
// "backward substitution"),
//   x_j = rho_j c_j + mu_j x_{j+off},   rho_j = 1/p_j,  mu_j = -q_j/p_j,
// a first-order linear recurrence.  On the GPU it is a scan of affine maps x -> m x + b
// (the multipliers kept as logs, so long products do not drift):
// each block reduces a tile of coefficients to one map per chain, a second kernel
// scans the tile maps of each vector, a third replays each tile from its carried-in value.
// The transposes (reverse mode) are (S^T g)_k = p_k g_k + q_{k-off} g_{k-off} and, for the
// inverse, the same recurrence run upward with mu'_k = -q_{k-off}/p_k.
//
// Diagonal scalings out = diag(s) A diag(sigma) (the Chebyshev normalisation of jac2cheb /
// cheb2jac) fold into the tables of the last / first factor.  Tables are float64 closed
// forms rounded once to the execute precision, so the kernels do no division.  All of this
// is ~3 flops per 8 bytes moved: bound by HBM.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "tdh_internal.cuh"

namespace tdh {
namespace {

constexpr int kThreads = 256;
constexpr int kTile = 2048;     // forward factors: coefficients per block
constexpr int kMaxM = 16;       // factors per step
constexpr int kInvRows = 5;     // table rows of an inverse factor
// back-substitution: E coefficients per thread (a tile of 4096 floats or 2048 doubles; the
// three staged arrays take 50 KB of dynamic shared memory), one padding slot per 128 bytes
template <typename T>
struct Scan {
    static constexpr int E = 64 / (int)sizeof(T);
    static constexpr int tile = kThreads * E;
    static constexpr int per_pad = 128 / (int)sizeof(T);
    static constexpr int smem = tile + tile / per_pad;
};

struct FactorSpec {
    int family;    // SP_ULTRA, SP_JACOBI, SP_IDENTITY
    int off;
    int M;
    int inverse;
    int flip;
    double par0, dir, b;
    int64_t n, ld;
};

__device__ void factor_pq(const FactorSpec& F, double par, int64_t j, double* p, double* q) {
    const double x = (double)j;
    if (F.family == SP_ULTRA) {
        *p = par / (par + x);
        *q = -par / (par + x + 2.0);
    } else if (F.family == SP_JACOBI) {
        const double s = par + F.b;
        *p = j == 0 ? 1.0 : (x + s + 1.0) / (2.0 * x + s + 1.0);
        *q = -(x + F.b + 1.0) / (2.0 * x + s + 3.0);
        if (F.flip) *q = -*q;
    } else {
        *p = 1.0;
        *q = 0.0;
    }
}

// 1 - mu_j for the downward recurrence (mu_j = -q_j/p_j) and 1 - mu'_k for the upward one
// (mu'_k = -q_{k-off}/p_k) of an unflipped, unscaled factor, in closed form (no cancellation
// near 1):  ultraspherical  1 - mu_j = 2/(l+j+2),  mu'_k = 1;
//           Jacobi          1 - mu_j = (2j(a+1) + (a+b+1)(a+2)) / ((2j+a+b+3)(j+a+b+1)),
//                           1 - mu_0 = (a+2)/(a+b+3),  1 - mu'_k = (a+1)/(k+a+b+1).
__device__ double delta_down(const FactorSpec& F, double par, int64_t j) {
    const double x = (double)j;
    if (F.family == SP_ULTRA) return 2.0 / (par + x + 2.0);
    if (F.family == SP_JACOBI) {
        const double a = par, s = par + F.b;
        if (j == 0) return (a + 2.0) / (s + 3.0);
        return (2.0 * x * (a + 1.0) + (s + 1.0) * (a + 2.0)) / ((2.0 * x + s + 3.0) * (x + s + 1.0));
    }
    return 1.0;
}

__device__ double delta_up(const FactorSpec& F, double par, int64_t k) {
    if (F.family == SP_ULTRA) return 0.0;
    if (F.family == SP_JACOBI) return (par + 1.0) / ((double)k + par + F.b + 1.0);
    return 1.0;
}

// forward: tab[f][0][j] = s_j p_j sigma_j, tab[f][1][j] = s_j q_j sigma_{j+off};
// inverse (tables of the unflipped factor; a flip is applied as signs by the kernels):
//   tab[f][0][j] = rho_j = s_j sigma_j / p_j,
//   tab[f][1][j] = delta_j = 1 - mu_j s_j / s_{j+off}  (downward recurrence, 1 past the end),
//   tab[f][2][j] = log(1 - delta_j)                       (-inf where the multiplier is 0),
//   tab[f][3][k] = 1 - mu'_k sigma_k / sigma_{k-off}    (upward recurrence, 1 for k < off),
//   tab[f][4][k] = its log;
// with a scale ratio r, 1 - mu r = (1 - r) + (1 - mu) r.  Every multiplier is positive.
// s = sout on the last factor, sigma = sin on the first, 1 elsewhere; zero for j >= n.
template <typename T>
__global__ void k_sparse_tables(FactorSpec F, const double* __restrict__ sout,
                                const double* __restrict__ sin, T* __restrict__ tab) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= F.ld * F.M) return;
    const int f = (int)(i / F.ld);
    const int64_t j = i % F.ld;
    const int rows = F.inverse ? kInvRows : 2;
    T* t = tab + (int64_t)f * rows * F.ld;
    if (j >= F.n) {
        for (int r = 0; r < rows; ++r) t[r * F.ld + j] = T(0);
        return;
    }
    const double par = F.par0 + F.dir * (double)f;
    const double* so = (f == F.M - 1) ? sout : nullptr;
    const double* si = (f == 0) ? sin : nullptr;
    auto S = [&](int64_t k) { return so ? so[k] : 1.0; };
    auto G = [&](int64_t k) { return si ? si[k] : 1.0; };
    double p, q;
    if (!F.inverse) {
        factor_pq(F, par, j, &p, &q);
        const bool up = j + F.off < F.n;
        t[j] = (T)(S(j) * p * G(j));
        t[F.ld + j] = up ? (T)(S(j) * q * G(j + F.off)) : T(0);
        return;
    }
    FactorSpec U = F;
    U.flip = 0;
    factor_pq(U, par, j, &p, &q);
    t[j] = (T)(S(j) * G(j) / p);
    double dn = 1.0, du = 1.0;
    if (j + F.off < F.n) {
        dn = delta_down(U, par, j);
        if (so) {
            const double r = S(j) / S(j + F.off);
            dn = (1.0 - r) + dn * r;
        }
    }
    if (j >= F.off) {
        du = delta_up(U, par, j);
        if (si) {
            const double r = G(j) / G(j - F.off);
            du = (1.0 - r) + du * r;
        }
    }
    t[F.ld + j] = (T)dn;
    t[2 * F.ld + j] = (T)log1p(-dn);
    t[3 * F.ld + j] = (T)du;
    t[4 * F.ld + j] = (T)log1p(-du);
}

// ---------------------------------------------------------------- forward factors

// Halo of each tile for an in-place step: the OFF*M coefficients after the tile (forward) or
// before it (transpose), saved before any block overwrites them.
template <typename T>
__global__ void k_halo_save(const T* __restrict__ x, T* __restrict__ halo, int64_t n,
                            int64_t ntiles, int H, int adjoint, int64_t total) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= total) return;
    const int64_t vt = i / H;
    const int e = (int)(i % H);
    const int64_t v = vt / ntiles, t = vt % ntiles;
    const int64_t j = adjoint ? t * kTile - H + e : (t + 1) * kTile + e;
    halo[i] = (j >= 0 && j < n) ? x[v * n + j] : T(0);
}

// Each block stages a tile plus a halo of OFF*M coefficients in shared memory and applies
// the M factors in turn (the halo shrinks by OFF per factor, so the tile stays exact).
template <typename T, int OFF>
__global__ void __launch_bounds__(kThreads) k_fwd_tile(const T* in, T* out, int64_t n,
                                                       int64_t ntiles, const T* __restrict__ tab,
                                                       int64_t ld, int M, int adjoint,
                                                       const T* __restrict__ halo) {
    __shared__ T buf[2][kTile + OFF * kMaxM];
    const int64_t vec = blockIdx.x / ntiles;
    const int64_t tile = blockIdx.x % ntiles;
    const int64_t j0 = tile * kTile;
    const T* x = in + vec * n;
    const int H = OFF * M;
    const int W = kTile + H;
    const int64_t base = adjoint ? j0 - H : j0;
    const T* hv = halo ? halo + (vec * ntiles + tile) * H : nullptr;
    for (int i = threadIdx.x; i < W; i += kThreads) {
        const int64_t j = base + i;
        T v = T(0);
        if (j >= 0 && j < n) {
            const bool in_halo = adjoint ? i < H : i >= kTile;
            v = (hv && in_halo) ? hv[adjoint ? i : i - kTile] : x[j];
        }
        buf[0][i] = v;
    }
    __syncthreads();
    int cur = 0;
    for (int f = 0; f < M; ++f) {
        const int ff = adjoint ? M - 1 - f : f;
        const T* P = tab + (int64_t)(2 * ff) * ld;
        const T* Q = P + ld;
        for (int i = threadIdx.x; i < W; i += kThreads) {
            const int64_t j = base + i;
            T v = T(0);
            if (j >= 0 && j < n) {
                if (!adjoint) {
                    const T c2 = (i + OFF < W) ? buf[cur][i + OFF] : T(0);
                    v = P[j] * buf[cur][i] + Q[j] * c2;
                } else {
                    const T g2 = (i >= OFF && j >= OFF) ? buf[cur][i - OFF] * Q[j - OFF] : T(0);
                    v = P[j] * buf[cur][i] + g2;
                }
            }
            buf[cur ^ 1][i] = v;
        }
        __syncthreads();
        cur ^= 1;
    }
    const int o = adjoint ? H : 0;
    T* y = out + vec * n;
    for (int i = threadIdx.x; i < kTile; i += kThreads) {
        const int64_t j = j0 + i;
        if (j < n) y[j] = buf[cur][i + o];
    }
}

// One factor, float32, n % 4 == 0, out of place: one float4 of a vector per thread, the
// neighbouring float4 supplies c_{j+off} (or g_{k-off}) from cache.
template <int OFF>
__global__ void __launch_bounds__(kThreads) k_fwd_f4(const float4* __restrict__ in,
                                                     float4* __restrict__ out, int64_t nq,
                                                     int64_t total, const float4* __restrict__ P4,
                                                     const float4* __restrict__ Q4, int adjoint) {
    const int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (c >= total) return;
    const int64_t q = c % nq;
    const float4 x = in[c];
    const float4 p = P4[q];
    float4 r;
    if (!adjoint) {
        const float4 qq = Q4[q];  // zero where j + off >= n
        const bool last = q + 1 == nq;
        const float4 xn = last ? make_float4(0.f, 0.f, 0.f, 0.f) : in[c + 1];
        if (OFF == 2) {
            r.x = p.x * x.x + qq.x * x.z;
            r.y = p.y * x.y + qq.y * x.w;
            r.z = p.z * x.z + qq.z * xn.x;
            r.w = p.w * x.w + qq.w * xn.y;
        } else {
            r.x = p.x * x.x + qq.x * x.y;
            r.y = p.y * x.y + qq.y * x.z;
            r.z = p.z * x.z + qq.z * x.w;
            r.w = p.w * x.w + qq.w * xn.x;
        }
    } else {
        const float4 qq = Q4[q];
        const bool first = q == 0;
        const float4 xp = first ? make_float4(0.f, 0.f, 0.f, 0.f) : in[c - 1];
        const float4 qp = first ? make_float4(0.f, 0.f, 0.f, 0.f) : Q4[q - 1];
        if (OFF == 2) {
            r.x = p.x * x.x + qp.z * xp.z;
            r.y = p.y * x.y + qp.w * xp.w;
            r.z = p.z * x.z + qq.x * x.x;
            r.w = p.w * x.w + qq.y * x.y;
        } else {
            r.x = p.x * x.x + qp.w * xp.w;
            r.y = p.y * x.y + qq.x * x.x;
            r.z = p.z * x.z + qq.y * x.y;
            r.w = p.w * x.w + qq.z * x.z;
        }
    }
    out[c] = r;
}

// ---------------------------------------------------------------- back-substitution

// Affine map x -> m x + b on each of the OFF interleaved chains, with the multiplier (always
// positive) kept as L = log m: composites add their logs, so a product over N positions
// carries O(log N) roundings.  Multiplying the rounded factors 1 - delta instead drifts by
// up to N ulp when the rounding errors are correlated, as they are for slowly varying
// multipliers near 1 (measured 5e-5 relative at n = 2^20 in float32).  Single positions use
// x - delta x, exact to the rounding of delta.
template <typename T, int OFF>
struct Aff {
    T L[OFF], b[OFF];
};

template <typename T, int OFF>
__device__ __forceinline__ Aff<T, OFF> aff_id() {
    Aff<T, OFF> r;
#pragma unroll
    for (int c = 0; c < OFF; ++c) {
        r.L[c] = T(0);
        r.b[c] = T(0);
    }
    return r;
}

// expm1(L) for |L| <= 1/2 by its Taylor series (float: degree 9, remainder below 2^-26 of
// the result); double uses the library function.
__device__ __forceinline__ float expm1_small(float L) {
    float t = 1.0f + L * (1.0f / 9.0f);
    t = 1.0f + L * (1.0f / 8.0f) * t;
    t = 1.0f + L * (1.0f / 7.0f) * t;
    t = 1.0f + L * (1.0f / 6.0f) * t;
    t = 1.0f + L * (1.0f / 5.0f) * t;
    t = 1.0f + L * (1.0f / 4.0f) * t;
    t = 1.0f + L * (1.0f / 3.0f) * t;
    t = 1.0f + L * 0.5f * t;
    return L * t;
}
__device__ __forceinline__ double expm1_small(double L) { return expm1(L); }

// exp(L) x: near m = 1 as x + expm1(L) x (relative accuracy of m - 1 kept)
template <typename T>
__device__ __forceinline__ T mul_m(T L, T x) {
    return L > T(-0.5) ? fma(expm1_small(L), x, x) : exp(L) * x;
}

// x first, then y
template <typename T, int OFF>
__device__ __forceinline__ Aff<T, OFF> aff_then(const Aff<T, OFF>& x, const Aff<T, OFF>& y) {
    Aff<T, OFF> r;
#pragma unroll
    for (int c = 0; c < OFF; ++c) {
        r.L[c] = x.L[c] + y.L[c];
        r.b[c] = mul_m(y.L[c], x.b[c]) + y.b[c];
    }
    return r;
}

template <typename T, int OFF>
__device__ __forceinline__ Aff<T, OFF> aff_shfl_up(const Aff<T, OFF>& v, int k) {
    Aff<T, OFF> r;
#pragma unroll
    for (int c = 0; c < OFF; ++c) {
        r.L[c] = __shfl_up_sync(0xffffffffu, v.L[c], k);
        r.b[c] = __shfl_up_sync(0xffffffffu, v.b[c], k);
    }
    return r;
}

// padded shared-memory slot: thread t reads slots E*t .. E*t+E-1 without bank conflicts
template <typename T>
__device__ __forceinline__ int spad(int i) { return i + i / Scan<T>::per_pad; }

// Exclusive block scan of the threads' maps (thread order); *total = all threads' map.
// warp_tot: [kThreads / 32 + 1] shared scratch.
template <typename T, int OFF>
__device__ Aff<T, OFF> block_exclusive(const Aff<T, OFF>& mine, Aff<T, OFF>* warp_tot,
                                       Aff<T, OFF>* total) {
    constexpr int NW = kThreads / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    Aff<T, OFF> inc = mine;
#pragma unroll
    for (int k = 1; k < 32; k <<= 1) {
        const Aff<T, OFF> o = aff_shfl_up(inc, k);
        if (lane >= k) inc = aff_then(o, inc);
    }
    Aff<T, OFF> exl = aff_shfl_up(inc, 1);
    if (lane == 0) exl = aff_id<T, OFF>();
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        // exclusive scan of the warp totals by the first warp; the total goes to slot NW
        Aff<T, OFF> v = lane < NW ? warp_tot[lane] : aff_id<T, OFF>();
#pragma unroll
        for (int k = 1; k < NW; k <<= 1) {
            const Aff<T, OFF> o = aff_shfl_up(v, k);
            if (lane >= k) v = aff_then(o, v);
        }
        Aff<T, OFF> ex = aff_shfl_up(v, 1);
        if (lane == 0) ex = aff_id<T, OFF>();
        __syncwarp();
        if (lane < NW) warp_tot[lane] = ex;
        if (lane == NW - 1) warp_tot[NW] = v;
    }
    __syncthreads();
    if (total) *total = warp_tot[NW];
    return aff_then(warp_tot[warp], exl);
}

// Logical position l runs in recurrence order: physical index l (REV = 0, x_k depends on
// x_{k-off}) or n-1-l (REV = 1, x_j depends on x_{j+off}).  Stages b = rho * c (times
// (-1)^j for a factor conjugated by diag((-1)^k)), delta = 1 - multiplier and log(multiplier)
// of each position of the tile; positions past the end are identity maps.
template <typename T, int REV>
__device__ void scan_load(const T* x, int64_t n, int64_t l0, const T* __restrict__ rho,
                          const T* __restrict__ delta, const T* __restrict__ logm, int flip,
                          T* sb, T* sd, T* sl) {
    constexpr int IT = Scan<T>::tile / kThreads, BATCH = 8;
    static_assert(IT % BATCH == 0, "load batches");
#pragma unroll
    for (int i0 = 0; i0 < IT; i0 += BATCH) {
        // all loads of a batch first (independent, in flight together), then the stores
        T bv[BATCH], dv[BATCH], lv[BATCH];
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int i = threadIdx.x + (i0 + u) * kThreads;
            const int64_t l = l0 + i;
            bv[u] = T(0);
            dv[u] = T(0);
            lv[u] = T(0);
            if (l < n) {
                const int64_t j = REV ? n - 1 - l : l;
                bv[u] = rho[j] * x[j];
                if (flip && (j & 1)) bv[u] = -bv[u];
                dv[u] = delta[j];
                lv[u] = logm[j];
            }
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            const int i = threadIdx.x + (i0 + u) * kThreads;
            sb[spad<T>(i)] = bv[u];
            sd[spad<T>(i)] = dv[u];
            sl[spad<T>(i)] = lv[u];
        }
    }
}

template <typename T, int OFF>
__device__ Aff<T, OFF> thread_map(const T* sb, const T* sd, const T* sl) {
    Aff<T, OFF> r = aff_id<T, OFF>();
#pragma unroll
    for (int e = 0; e < Scan<T>::E; ++e) {
        const int i = spad<T>(threadIdx.x * Scan<T>::E + e);
        const int c = e % OFF;
        r.L[c] += sl[i];
        r.b[c] = fma(-sd[i], r.b[c], r.b[c]) + sb[i];
    }
    return r;
}

// Kernel 1: the map of every tile (its chains' values at the tile end as functions of the
// values entering it).  sum: [batch * ntiles] maps.
template <typename T, int OFF, int REV>
__global__ void __launch_bounds__(kThreads) k_scan_tiles(const T* __restrict__ in, int64_t n,
                                                         int64_t ntiles, const T* __restrict__ rho,
                                                         const T* __restrict__ delta,
                                                         const T* __restrict__ logm, int flip,
                                                         Aff<T, OFF>* __restrict__ sum) {
    extern __shared__ __align__(16) unsigned char scan_smem[];
    T* sb = reinterpret_cast<T*>(scan_smem);
    T* sd = sb + Scan<T>::smem;
    T* sl = sd + Scan<T>::smem;
    __shared__ Aff<T, OFF> wt[kThreads / 32 + 1];
    const int64_t vec = blockIdx.x / ntiles, tile = blockIdx.x % ntiles;
    scan_load<T, REV>(in + vec * n, n, tile * Scan<T>::tile, rho, delta, logm, flip, sb, sd, sl);
    __syncthreads();
    const Aff<T, OFF> mine = thread_map<T, OFF>(sb, sd, sl);
    Aff<T, OFF> tot;
    block_exclusive<T, OFF>(mine, wt, &tot);
    if (threadIdx.x == 0) sum[blockIdx.x] = tot;
}

// Kernel 2: per vector, the values entering each tile (x = 0 before the first position).
template <typename T, int OFF>
__global__ void __launch_bounds__(kThreads) k_scan_carry(const Aff<T, OFF>* __restrict__ sum,
                                                         int64_t ntiles,
                                                         Aff<T, OFF>* __restrict__ carry) {
    __shared__ Aff<T, OFF> wt[kThreads / 32 + 1];
    const Aff<T, OFF>* s = sum + (int64_t)blockIdx.x * ntiles;
    Aff<T, OFF>* cr = carry + (int64_t)blockIdx.x * ntiles;
    const int64_t per = (ntiles + kThreads - 1) / kThreads;
    const int64_t t0 = std::min<int64_t>(ntiles, per * threadIdx.x);
    const int64_t t1 = std::min<int64_t>(ntiles, t0 + per);
    Aff<T, OFF> mine = aff_id<T, OFF>();
    for (int64_t t = t0; t < t1; ++t) mine = aff_then(mine, s[t]);
    Aff<T, OFF> run = block_exclusive<T, OFF>(mine, wt, nullptr);
    for (int64_t t = t0; t < t1; ++t) {
        cr[t] = run;  // entering values = run.b (run applied to 0)
        run = aff_then(run, s[t]);
    }
}

// Kernel 3: replay each tile from its entering values and write x (in place allowed: a
// block reads its whole tile before writing it).
template <typename T, int OFF, int REV>
__global__ void __launch_bounds__(kThreads) k_scan_solve(const T* in, T* out, int64_t n,
                                                         int64_t ntiles, const T* __restrict__ rho,
                                                         const T* __restrict__ delta,
                                                         const T* __restrict__ logm, int flip,
                                                         const Aff<T, OFF>* __restrict__ carry) {
    extern __shared__ __align__(16) unsigned char scan_smem[];
    T* sb = reinterpret_cast<T*>(scan_smem);
    T* sd = sb + Scan<T>::smem;
    T* sl = sd + Scan<T>::smem;
    __shared__ Aff<T, OFF> wt[kThreads / 32 + 1];
    const int64_t vec = blockIdx.x / ntiles, tile = blockIdx.x % ntiles;
    const int64_t l0 = tile * Scan<T>::tile;
    scan_load<T, REV>(in + vec * n, n, l0, rho, delta, logm, flip, sb, sd, sl);
    __syncthreads();
    const Aff<T, OFF> mine = thread_map<T, OFF>(sb, sd, sl);
    const Aff<T, OFF> ex = block_exclusive<T, OFF>(mine, wt, nullptr);
    const Aff<T, OFF> cin = carry[blockIdx.x];
    T st[OFF];
#pragma unroll
    for (int c = 0; c < OFF; ++c) st[c] = mul_m(ex.L[c], cin.b[c]) + ex.b[c];
#pragma unroll
    for (int e = 0; e < Scan<T>::E; ++e) {
        const int i = spad<T>(threadIdx.x * Scan<T>::E + e);
        const int c = e % OFF;
        st[c] = fma(-sd[i], st[c], st[c]) + sb[i];
        sb[i] = st[c];
    }
    __syncthreads();
    T* y = out + vec * n;
    for (int i = threadIdx.x; i < Scan<T>::tile; i += kThreads) {
        const int64_t l = l0 + i;
        if (l < n) {
            const int64_t j = REV ? n - 1 - l : l;
            const T v = sb[spad<T>(i)];
            y[j] = (flip && (j & 1)) ? -v : v;
        }
    }
}

// ------------------------------------------------- back-substitution as a weighted prefix sum
//
// With W the solution of the homogeneous recurrence, W_j = mu_j W_{j+off}, the inverse factor is
//   x_j = W_j sum_{i >= j, i = j mod off} U_i c_i,   U = rho / W,
// (and its transpose x_i = U_i sum_{j <= i} W_j g_j): a plain sum per chain between two
// products, where the affine scan above carries a multiplier.  W and U are closed forms:
//   ultraspherical  W_j = (l + j) / l,                              U_j = 1 / (p_j W_j) = 1;
//   Jacobi          W_j = (2j+s+1) Gamma(j+s+1) / Gamma(j+b+1),     U_j = 1 / (p_j W_j),  s = a+b
// (W_0 = mu_0 W_1), scaled so that the smallest W is 1; signs of a flipped factor and the diagonal
// scalings fold into them.  A suffix sum is then x_j / W_j <= x_j, a term U_i c_i the difference of
// two of them, so nothing overflows before the result does (times two).  In the transpose the
// prefix sums are x_i / U_i, so there W comes down, and U goes up, by a power of two (sp_gain) that
// makes the smallest U about 1.  U falls to about 1 / W:
// terms below the type's least normal value lose digits that only matter to results as small,
// so they are taken where ln W spans at most sum_range (float32: 24, full precision down to inputs
// of 2^-91; parameters a below 0.7 at n = 2^20, 1.1 at 2^16), and the affine scan stays for larger
// parameters.  (Ultraspherical: any range.)
//
// Precision.  A single factor sums in its own precision (log2 n roundings per sum instead of n).
// Float32 chains of several factors or steps amplify what one inverse leaves behind (a factor
// sums its predecessor's errors over the whole tail), so there the tables, the sums and the
// values between consecutive inverse factors are pairs of floats (FF, about 44 bits), rounded
// once at the end; float64 chains keep the affine scan.
//
// Bound by HBM: k_sum_tiles reads the vectors once (tile sums), k_sum_solve reads them again,
// from L2 when the batch fits, and writes the result; it also forms the tile sums the next
// factor needs.  16 x 2^20 float32, C^(1.25) -> C^(0.25): 46 us against 140 us for the three
// kernels of the affine scan (a plain copy of the batch: 20 us); two factors in pairs of
// floats, C^(2.25) -> C^(0.25): 216 against 277 us.
constexpr double sum_range(int prec) { return prec == TDH_FP64 ? 40.0 : 24.0; }
constexpr int kSumChunks = 4;  // pieces per thread

// A pair of floats h + l, |l| <= ulp(h) / 2 (Dekker 1971; Knuth's two-sum).
struct __align__(8) FF {
    float h, l;
};
__device__ __forceinline__ FF ff_fast(float a, float b) {
    const float s = __fadd_rn(a, b);
    return FF{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ FF add(FF a, FF b) {
    const float s = __fadd_rn(a.h, b.h), bb = __fsub_rn(s, a.h);
    const float e = __fadd_rn(__fsub_rn(a.h, __fsub_rn(s, bb)), __fsub_rn(b.h, bb));
    return ff_fast(s, __fadd_rn(e, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ FF mul(FF a, float b) {
    const float p = __fmul_rn(a.h, b);
    return ff_fast(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ FF mul(FF a, FF b) {
    const float p = __fmul_rn(a.h, b.h);
    return ff_fast(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ float mul(float a, float b) { return a * b; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ void put(float& o, float v) { o = v; }
__device__ __forceinline__ void put(double& o, double v) { o = v; }
__device__ __forceinline__ void put(float& o, FF v) { o = v.h; }
__device__ __forceinline__ void put(FF& o, FF v) { o = v; }
__device__ __forceinline__ void from_double(float& o, double v) { o = (float)v; }
__device__ __forceinline__ void from_double(double& o, double v) { o = v; }
__device__ __forceinline__ void from_double(FF& o, double v) {
    o.h = (float)v;
    o.l = isfinite(o.h) ? (float)(v - (double)o.h) : 0.0f;
}
// v times a power of two
__device__ __forceinline__ float scaled(float v, float g) { return v * g; }
__device__ __forceinline__ double scaled(double v, float g) { return v * (double)g; }
__device__ __forceinline__ FF scaled(FF v, float g) { return FF{v.h * g, v.l * g}; }
template <bool DOWN, typename A>
__device__ __forceinline__ A shfl_by(A v, int d) {
    if constexpr (std::is_same<A, FF>::value)
        return FF{shfl_by<DOWN>(v.h, d), shfl_by<DOWN>(v.l, d)};
    else
        return DOWN ? __shfl_down_sync(0xffffffffu, v, d) : __shfl_up_sync(0xffffffffu, v, d);
}
template <typename A>
__device__ __forceinline__ A shfl_at(A v, int lane) {
    if constexpr (std::is_same<A, FF>::value)
        return FF{shfl_at(v.h, lane), shfl_at(v.l, lane)};
    else
        return __shfl_sync(0xffffffffu, v, lane);
}

// A: type of the sums and tables; V coefficients per piece.
template <typename A>
struct SumTile {
    static constexpr int V = std::is_same<A, double>::value ? 2 : 4;
    static constexpr int chunk = kThreads * V;
    static constexpr int tile = kSumChunks * chunk;
};

// V consecutive values at j (ALIGNED: n a multiple of V, 16-byte accesses), 0 past n
template <int V, bool ALIGNED, typename X>
__device__ __forceinline__ void load_piece(const X* p, int64_t j, int64_t n, X (&v)[V]) {
    if constexpr (ALIGNED) {
        constexpr int W = (int)(V * sizeof(X) / 4);
        float* f = reinterpret_cast<float*>(v);
        if (j < n) {
            const float* q = reinterpret_cast<const float*>(p + j);
#pragma unroll
            for (int i = 0; i < W; i += 4) {
                const float4 t = *reinterpret_cast<const float4*>(q + i);
                f[i] = t.x, f[i + 1] = t.y, f[i + 2] = t.z, f[i + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < W; ++i) f[i] = 0.0f;
        }
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = j + i < n ? p[j + i] : X{};
    }
}
template <int V, bool ALIGNED, typename X>
__device__ __forceinline__ void store_piece(X* p, int64_t j, int64_t n, const X (&v)[V]) {
    if constexpr (ALIGNED) {
        constexpr int W = (int)(V * sizeof(X) / 4);
        const float* f = reinterpret_cast<const float*>(v);
        if (j < n) {
            float* q = reinterpret_cast<float*>(p + j);
#pragma unroll
            for (int i = 0; i < W; i += 4)
                *reinterpret_cast<float4*>(q + i) = make_float4(f[i], f[i + 1], f[i + 2], f[i + 3]);
        }
    } else {
#pragma unroll
        for (int i = 0; i < V; ++i)
            if (j + i < n) p[j + i] = v[i];
    }
}

template <typename A, int OFF>
struct ChainSum {
    A v[OFF];
};

// Sum over the block, the same in every thread (fixed order); red: [kThreads / 32] slots.
template <typename A, int OFF>
__device__ __forceinline__ ChainSum<A, OFF> block_sum(ChainSum<A, OFF> x, ChainSum<A, OFF>* red) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1)
#pragma unroll
        for (int c = 0; c < OFF; ++c) x.v[c] = add(x.v[c], shfl_at(x.v[c], lane ^ k));
    if (lane == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    ChainSum<A, OFF> t = red[0];
#pragma unroll
    for (int w = 1; w < kThreads / 32; ++w)
#pragma unroll
        for (int c = 0; c < OFF; ++c) t.v[c] = add(t.v[c], red[w].v[c]);
    return t;
}

// sum[v ntiles + t]: per chain (j mod OFF), the sum of weight_j in_j over tile t (GAIN: the weights
// times gain).
template <typename A, typename TI, int OFF, bool GAIN, bool ALIGNED>
__global__ void __launch_bounds__(kThreads) k_sum_tiles(const TI* __restrict__ in, int64_t n,
                                                        int64_t ntiles,
                                                        const A* __restrict__ weight, float gain,
                                                        ChainSum<A, OFF>* __restrict__ sum) {
    constexpr int V = SumTile<A>::V;
    __shared__ ChainSum<A, OFF> red[kThreads / 32];
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t vec = blockIdx.x / ntiles, tile = blockIdx.x % ntiles;
    const TI* x = in + vec * n;
    ChainSum<A, OFF> s{};
    TI xv[kSumChunks][V];
    A wv[kSumChunks][V];
#pragma unroll
    for (int k = 0; k < kSumChunks; ++k) {
        const int64_t j = tile * SumTile<A>::tile + k * SumTile<A>::chunk + threadIdx.x * V;
        load_piece<V, ALIGNED>(x, j, n, xv[k]);
        load_piece<V, ALIGNED>(weight, j, n, wv[k]);
    }
#pragma unroll
    for (int k = 0; k < kSumChunks; ++k)
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const A w = GAIN ? scaled(wv[k][i], gain) : wv[k][i];
            s.v[i % OFF] = add(s.v[i % OFF], mul(w, xv[k][i]));
        }
    s = block_sum<A, OFF>(s, red);
    if (threadIdx.x == 0) sum[blockIdx.x] = s;
}

// sum[v ntiles + t] <- the sum of the tiles after (REV) or before t: where a vector has many tiles,
// adding them up in every block would be quadratic in n (2^27 coefficients: as many bytes as the
// vector's).  One block per vector, a thread takes a strip of tiles.  Float32 C^(1.25) -> C^(0.25):
// 2^27 690 -> 600 us, 2^29 5.7 -> 2.3 ms, two factors 24 -> 8.4 ms (affine scan 5.5 and 11 ms); at
// 4 x 2^24 it costs as much as it saves (269 and 261 us).
constexpr int kCarryTiles = 4097;  // tiles of a vector from which this pays
template <typename A, int OFF, bool REV>
__global__ void __launch_bounds__(kThreads) k_sum_carry(ChainSum<A, OFF>* __restrict__ sum,
                                                        int64_t ntiles) {
    __shared__ ChainSum<A, OFF> tot[kThreads];
    ChainSum<A, OFF>* s = sum + (int64_t)blockIdx.x * ntiles;
    const int64_t per = (ntiles + kThreads - 1) / kThreads;
    const int64_t t0 = min((int64_t)threadIdx.x * per, ntiles), t1 = min(t0 + per, ntiles);
    ChainSum<A, OFF> mine{};
    for (int64_t t = t0; t < t1; ++t)
#pragma unroll
        for (int c = 0; c < OFF; ++c) mine.v[c] = add(mine.v[c], s[t].v[c]);
    // inclusive scan of the strips, in the direction of the sums
    const int at = REV ? kThreads - 1 - (int)threadIdx.x : (int)threadIdx.x;
    tot[at] = mine;
    __syncthreads();
    for (int d = 1; d < kThreads; d <<= 1) {
        const ChainSum<A, OFF> o = at >= d ? tot[at - d] : ChainSum<A, OFF>{};
        __syncthreads();
#pragma unroll
        for (int c = 0; c < OFF; ++c) tot[at].v[c] = add(tot[at].v[c], o.v[c]);
        __syncthreads();
    }
    ChainSum<A, OFF> run = at > 0 ? tot[at - 1] : ChainSum<A, OFF>{};
    for (int64_t i = 0; i < t1 - t0; ++i) {
        const int64_t t = REV ? t1 - 1 - i : t0 + i;
        const ChainSum<A, OFF> x = s[t];
        s[t] = run;
#pragma unroll
        for (int c = 0; c < OFF; ++c) run.v[c] = add(run.v[c], x.v[c]);
    }
}

// out_j = wout_j (sum over the chain of win_i in_i, i >= j (REV) or i <= j); then, where `next` is
// given, the tile sums of next_j out_j.  The block's carry is the sum of the tiles after (before)
// its own, added in a fixed order (carried: sum holds it).  In place allowed: a block reads its tile before writing it.
// `first`: the input is older than the previous kernel, so it may be read before waiting for it.
// gain, next_gain: the transpose's powers of two on win and next (wout's is 1 / gain).
template <typename A, typename TI, typename TO, int OFF, bool REV, bool ALIGNED>
__global__ void __launch_bounds__(kThreads) k_sum_solve(const TI* in, TO* out, int64_t n,
                                                        int64_t ntiles, const A* __restrict__ win,
                                                        const A* __restrict__ wout,
                                                        const ChainSum<A, OFF>* sum,
                                                        const A* __restrict__ next,
                                                        ChainSum<A, OFF>* next_sum, int first,
                                                        float gain, float next_gain,
                                                        int carried) {
    constexpr int V = SumTile<A>::V;
    constexpr int NW = kThreads / 32;
    __shared__ ChainSum<A, OFF> red[NW], part[kSumChunks * NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int64_t vec = blockIdx.x / ntiles, tile = blockIdx.x % ntiles;
    const TI* x = in + vec * n;
    if (!first) asm volatile("griddepcontrol.wait;" ::: "memory");
    A v[kSumChunks][V];
    {
        TI xv[kSumChunks][V];
        A w[kSumChunks][V];
#pragma unroll
        for (int k = 0; k < kSumChunks; ++k) {
            const int64_t j = tile * SumTile<A>::tile + k * SumTile<A>::chunk + tid * V;
            load_piece<V, ALIGNED>(x, j, n, xv[k]);
            load_piece<V, ALIGNED>(win, j, n, w[k]);
        }
        // within a thread, in the direction of the sums
#pragma unroll
        for (int k = 0; k < kSumChunks; ++k) {
#pragma unroll
            for (int i = 0; i < V; ++i)
                v[k][i] = mul(REV ? w[k][i] : scaled(w[k][i], gain), xv[k][i]);
            if constexpr (REV) {
#pragma unroll
                for (int i = V - 1 - OFF; i >= 0; --i) v[k][i] = add(v[k][i], v[k][i + OFF]);
            } else {
#pragma unroll
                for (int i = OFF; i < V; ++i) v[k][i] = add(v[k][i], v[k][i - OFF]);
            }
        }
    }
    // exclusive scan of the threads' totals over the warp, per piece
    ChainSum<A, OFF> before[kSumChunks];
#pragma unroll
    for (int k = 0; k < kSumChunks; ++k) {
        ChainSum<A, OFF> s;
#pragma unroll
        for (int c = 0; c < OFF; ++c) s.v[c] = REV ? v[k][c] : v[k][V - OFF + c];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1)
#pragma unroll
            for (int c = 0; c < OFF; ++c) {
                const A o = shfl_by<REV>(s.v[c], d);
                if (REV ? lane + d < 32 : lane >= d) s.v[c] = add(s.v[c], o);
            }
        if (lane == (REV ? 0 : 31)) part[k * NW + warp] = s;
#pragma unroll
        for (int c = 0; c < OFF; ++c) {
            const A o = shfl_by<REV>(s.v[c], 1);
            before[k].v[c] = lane == (REV ? 31 : 0) ? A{} : o;
        }
    }
    if (first) asm volatile("griddepcontrol.wait;" ::: "memory");
    // the other tiles' sums
    ChainSum<A, OFF> carry{};
    if (carried && tid == 0) carry = sum[blockIdx.x];
    for (int64_t t = carried ? ntiles : (REV ? tile + 1 : 0) + tid; t < (REV ? ntiles : tile);
         t += kThreads)
#pragma unroll
        for (int c = 0; c < OFF; ++c) carry.v[c] = add(carry.v[c], sum[vec * ntiles + t].v[c]);
    carry = block_sum<A, OFF>(carry, red);  // its barrier also publishes `part`
    // the block's (piece, warp) totals that come first: one scan of 32 values per warp
    static_assert(kSumChunks * NW == 32, "one warp scans the block's totals");
    {
        ChainSum<A, OFF> s = part[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1)
#pragma unroll
            for (int c = 0; c < OFF; ++c) {
                const A o = shfl_by<REV>(s.v[c], d);
                if (REV ? lane + d < 32 : lane >= d) s.v[c] = add(s.v[c], o);
            }
#pragma unroll
        for (int k = 0; k < kSumChunks; ++k) {
            const int at = k * NW + warp + (REV ? 1 : -1);  // inclusive total just before
#pragma unroll
            for (int c = 0; c < OFF; ++c) {
                const A o = shfl_at(s.v[c], at & 31);
                before[k].v[c] = add(before[k].v[c], carry.v[c]);
                if (at >= 0 && at < 32) before[k].v[c] = add(before[k].v[c], o);
            }
        }
    }
    TO* y = out + vec * n;
    ChainSum<A, OFF> ns{};
#pragma unroll
    for (int k = 0; k < kSumChunks; ++k) {
        const int64_t j = tile * SumTile<A>::tile + k * SumTile<A>::chunk + tid * V;
        A o[V];
        load_piece<V, ALIGNED>(wout, j, n, o);
#pragma unroll
        for (int i = 0; i < V; ++i)
            o[i] = mul(REV ? o[i] : scaled(o[i], 1.0f / gain), add(v[k][i], before[k].v[i % OFF]));
        if (next) {
            A nw[V];
            load_piece<V, ALIGNED>(next, j, n, nw);
#pragma unroll
            for (int i = 0; i < V; ++i)
                ns.v[i % OFF] =
                    add(ns.v[i % OFF], mul(REV ? nw[i] : scaled(nw[i], next_gain), o[i]));
        }
        TO t[V];
#pragma unroll
        for (int i = 0; i < V; ++i) put(t[i], o[i]);
        store_piece<V, ALIGNED>(y, j, n, t);
    }
    if (next) {
        __syncthreads();  // every thread has read `red`
        ns = block_sum<A, OFF>(ns, red);
        if (tid == 0) next_sum[blockIdx.x] = ns;
    }
}

// tab[f][0][j] = s_j W_j, tab[f][1][j] = U_j sigma_j of factor f (signs of a flipped factor
// included); g: Gamma(j+s+1) / Gamma(j+b+1) (Jacobi), scale: W's normalisation.
template <typename A>
__global__ void k_sum_tables(FactorSpec F, int f, const double* __restrict__ g, double scale,
                             const double* __restrict__ sout, const double* __restrict__ sin,
                             A* __restrict__ tab) {
    const int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (j >= F.ld) return;
    A* t = tab + (int64_t)f * 2 * F.ld;
    if (j >= F.n) {
        t[j] = t[F.ld + j] = A{};
        return;
    }
    const double par = F.par0 + F.dir * (double)f, x = (double)j, s = par + F.b;
    FactorSpec U = F;
    U.flip = 0;
    double p, q, W;
    factor_pq(U, par, j, &p, &q);
    if (F.family == SP_ULTRA) {
        W = (par + x) / par;  // U = 1
    } else if (j == 0) {
        W = -q / p * (s + 3.0) * g[1] * scale;  // mu_0 W_1
    } else {
        W = (2.0 * x + s + 1.0) * g[j] * scale;
    }
    const double sign = (F.flip && (j & 1)) ? -1.0 : 1.0;
    const double so = f == F.M - 1 && sout ? sout[j] : 1.0;
    const double si = f == 0 && sin ? sin[j] : 1.0;
    from_double(t[j], so * W * sign);
    from_double(t[F.ld + j], sign * si * (F.family == SP_ULTRA ? 1.0 : 1.0 / (p * W)));
}

unsigned blocks_for(int64_t count) { return (unsigned)((count + kThreads - 1) / kThreads); }

template <typename T, int OFF>
int forward_typed(const Step& st, const void* in, void* out, int64_t batch, int adjoint,
                  cudaStream_t s) {
    const int64_t n = st.n;
    const T* tab = static_cast<const T*>(st.sp_tab);
    const bool inplace = in == out;
    if (std::is_same<T, float>::value && st.sp_M == 1 && n % 4 == 0 && !inplace) {
        const int64_t total = batch * (n / 4);
        k_fwd_f4<OFF><<<blocks_for(total), kThreads, 0, s>>>(
            static_cast<const float4*>(in), static_cast<float4*>(out), n / 4, total,
            reinterpret_cast<const float4*>(tab), reinterpret_cast<const float4*>(tab + st.sp_ld),
            adjoint);
        TDH_CUDA(cudaGetLastError());
        note_launches(1);
        return TDH_OK;
    }
    const int64_t ntiles = (n + kTile - 1) / kTile;
    const int H = OFF * st.sp_M;
    T* halo = nullptr;
    if (inplace) {
        const int64_t total = batch * ntiles * H;
        TDH_TRY(scratch_alloc(reinterpret_cast<void**>(&halo), sizeof(T) * total, s));
        k_halo_save<T><<<blocks_for(total), kThreads, 0, s>>>(static_cast<const T*>(in), halo, n,
                                                               ntiles, H, adjoint, total);
        note_launches(1);
    }
    k_fwd_tile<T, OFF><<<(unsigned)(batch * ntiles), kThreads, 0, s>>>(
        static_cast<const T*>(in), static_cast<T*>(out), n, ntiles, tab, st.sp_ld, st.sp_M,
        adjoint, halo);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) note_launches(1);
    if (halo) scratch_free(halo, s);
    TDH_CUDA(e);
    return TDH_OK;
}

template <typename T, int OFF>
int inverse_typed(const Step& st, const void* in, void* out, int64_t batch, int adjoint,
                  cudaStream_t s) {
    const int64_t n = st.n;
    const int64_t ntiles = (n + Scan<T>::tile - 1) / Scan<T>::tile;
    using A = Aff<T, OFF>;
    constexpr size_t smem = 3 * sizeof(T) * (size_t)Scan<T>::smem;
    static PerDevice attr_once;
    const cudaError_t attr = per_device(attr_once, [](int*) {
        const void* ks[4] = {(const void*)k_scan_tiles<T, OFF, 0>, (const void*)k_scan_tiles<T, OFF, 1>,
                             (const void*)k_scan_solve<T, OFF, 0>, (const void*)k_scan_solve<T, OFF, 1>};
        cudaError_t e = cudaSuccess;
        for (const void* k : ks)
            if (e == cudaSuccess)
                e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        return e;
    });
    if (attr != cudaSuccess) {
        set_error("cudaFuncSetAttribute: %s", cudaGetErrorString(attr));
        return TDH_ERR_CUDA;
    }
    A *sum = nullptr, *carry = nullptr;
    TDH_TRY(scratch_alloc(reinterpret_cast<void**>(&sum), sizeof(A) * batch * ntiles * 2, s));
    carry = sum + batch * ntiles;
    const unsigned grid = (unsigned)(batch * ntiles);
    cudaError_t e = cudaSuccess;
    for (int f = 0; f < st.sp_M && e == cudaSuccess; ++f) {
        // A^{-1} applies the factors' inverses in order; its transpose in reverse order
        const int ff = adjoint ? st.sp_M - 1 - f : f;
        const T* tab = static_cast<const T*>(st.sp_tab) + (int64_t)ff * kInvRows * st.sp_ld;
        const T* rho = tab;
        const T* src = static_cast<const T*>(f == 0 ? in : out);
        const int flip = st.sp_flip;
        if (!adjoint) {
            const T* dl = tab + st.sp_ld;
            const T* lg = tab + 2 * st.sp_ld;
            k_scan_tiles<T, OFF, 1><<<grid, kThreads, smem, s>>>(src, n, ntiles, rho, dl, lg, flip, sum);
            k_scan_carry<T, OFF><<<(unsigned)batch, kThreads, 0, s>>>(sum, ntiles, carry);
            k_scan_solve<T, OFF, 1><<<grid, kThreads, smem, s>>>(src, static_cast<T*>(out), n, ntiles,
                                                              rho, dl, lg, flip, carry);
        } else {
            const T* dl = tab + 3 * st.sp_ld;
            const T* lg = tab + 4 * st.sp_ld;
            k_scan_tiles<T, OFF, 0><<<grid, kThreads, smem, s>>>(src, n, ntiles, rho, dl, lg, flip, sum);
            k_scan_carry<T, OFF><<<(unsigned)batch, kThreads, 0, s>>>(sum, ntiles, carry);
            k_scan_solve<T, OFF, 0><<<grid, kThreads, smem, s>>>(src, static_cast<T*>(out), n, ntiles,
                                                              rho, dl, lg, flip, carry);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) note_launches(3);
    }
    scratch_free(sum, s);
    TDH_CUDA(e);
    return TDH_OK;
}

// in: TI, out: TO, the values between the step's own factors: M (all may share one buffer when
// they are of one type; `mid` otherwise).
template <typename A, typename TI, typename TO, typename M, int OFF, bool REV, bool ALIGNED>
int sums_typed(const Step& st, const void* in, void* out, int64_t batch, cudaStream_t s) {
    using S = ChainSum<A, OFF>;
    const int64_t n = st.n, ntiles = (n + SumTile<A>::tile - 1) / SumTile<A>::tile;
    const unsigned grid = (unsigned)(batch * ntiles);
    // two sets of tile sums: a factor reads one while it writes the next factor's
    const size_t sum_bytes = (sizeof(S) * 2 * (size_t)grid + 255) / 256 * 256;
    const bool own_mid = st.sp_M > 1 && !std::is_same<M, TO>::value;
    char* scr = nullptr;
    TDH_TRY(scratch_alloc(reinterpret_cast<void**>(&scr),
                          sum_bytes + (own_mid ? sizeof(M) * (size_t)(batch * n) : 0), s));
    S* sum = reinterpret_cast<S*>(scr);
    M* mid = own_mid ? reinterpret_cast<M*>(scr + sum_bytes) : static_cast<M*>(out);
    // A^{-1} applies the factors' inverses in order; its transpose (REV = false) in reverse
    auto row = [&](int f, int second) {
        const int ff = REV ? f : st.sp_M - 1 - f;
        return static_cast<const A*>(st.sp_tab) + ((int64_t)ff * 2 + second) * st.sp_ld;
    };
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    const int carried = ntiles >= kCarryTiles;
    auto gain = [&](int f) { return st.sp_gain[REV ? f : st.sp_M - 1 - f]; };
    cudaError_t e =
        cudaLaunchKernelEx(&cfg, k_sum_tiles<A, TI, OFF, !REV, ALIGNED>,
                           static_cast<const TI*>(in), n, ntiles, row(0, REV), gain(0), sum);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    for (int f = 0; f < st.sp_M && e == cudaSuccess; ++f) {
        const bool first = f == 0, last = f + 1 == st.sp_M;
        const A* next = last ? nullptr : row(f + 1, REV);
        const S* from = sum + (f & 1) * (size_t)grid;
        S* to = sum + ((f + 1) & 1) * (size_t)grid;
        const float g = gain(f), ng = last ? 1.0f : gain(f + 1);
        if (carried) {
            cfg.gridDim = dim3((unsigned)batch);
            cfg.numAttrs = 0;
            e = cudaLaunchKernelEx(&cfg, k_sum_carry<A, OFF, REV>, sum + (f & 1) * (size_t)grid,
                                   ntiles);
            cfg.gridDim = dim3(grid);
            cfg.numAttrs = 1;
            if (e != cudaSuccess) break;
        }
        if (first && last)
            e = cudaLaunchKernelEx(&cfg, k_sum_solve<A, TI, TO, OFF, REV, ALIGNED>,
                                   static_cast<const TI*>(in), static_cast<TO*>(out), n, ntiles,
                                   row(f, REV), row(f, !REV), from, next, to, 1, g, ng, carried);
        else if (first)
            e = cudaLaunchKernelEx(&cfg, k_sum_solve<A, TI, M, OFF, REV, ALIGNED>,
                                   static_cast<const TI*>(in), mid, n, ntiles, row(f, REV),
                                   row(f, !REV), from, next, to, 1, g, ng, carried);
        else if (last)
            e = cudaLaunchKernelEx(&cfg, k_sum_solve<A, M, TO, OFF, REV, ALIGNED>,
                                   (const M*)mid, static_cast<TO*>(out), n, ntiles, row(f, REV),
                                   row(f, !REV), from, next, to, 0, g, ng, carried);
        else
            e = cudaLaunchKernelEx(&cfg, k_sum_solve<A, M, M, OFF, REV, ALIGNED>, (const M*)mid,
                                   mid, n, ntiles, row(f, REV), row(f, !REV), from, next, to, 0, g, ng, carried);
    }
    scratch_free(scr, s);
    if (e != cudaSuccess) {
        set_error("back-substitution: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1 + (carried ? 2 : 1) * st.sp_M);
    return TDH_OK;
}

template <typename A, typename TI, typename TO, typename M, int OFF>
int sums_launch(const Step& st, const void* in, void* out, int64_t batch, int adjoint,
                cudaStream_t s) {
    // 16-byte accesses: rows of the vectors and of the tables (ld a multiple of four) aligned
    const bool al = st.n % SumTile<A>::V == 0 && (((uintptr_t)in | (uintptr_t)out) & 15) == 0;
    if (adjoint)
        return al ? sums_typed<A, TI, TO, M, OFF, false, true>(st, in, out, batch, s)
                  : sums_typed<A, TI, TO, M, OFF, false, false>(st, in, out, batch, s);
    return al ? sums_typed<A, TI, TO, M, OFF, true, true>(st, in, out, batch, s)
              : sums_typed<A, TI, TO, M, OFF, true, false>(st, in, out, batch, s);
}

// The step's sums: wide_in / wide_out say that in / out hold pairs of floats (between consecutive
// inverse steps of a float32 chain).
template <typename T, int OFF>
int sums_dispatch(const Step& st, const void* in, void* out, int64_t batch, int adjoint,
                  bool wide_in, bool wide_out, cudaStream_t s) {
    if constexpr (std::is_same<T, float>::value) {
        if (st.sp_sums == 2) {
            if (wide_in && wide_out)
                return sums_launch<FF, FF, FF, FF, OFF>(st, in, out, batch, adjoint, s);
            if (wide_in)
                return sums_launch<FF, FF, float, FF, OFF>(st, in, out, batch, adjoint, s);
            if (wide_out)
                return sums_launch<FF, float, FF, FF, OFF>(st, in, out, batch, adjoint, s);
            return sums_launch<FF, float, float, FF, OFF>(st, in, out, batch, adjoint, s);
        }
    }
    return sums_launch<T, T, T, T, OFF>(st, in, out, batch, adjoint, s);
}

template <typename T>
int launch_typed(const Step& st, const void* in, void* out, int64_t batch, int adjoint,
                 bool wide_in, bool wide_out, cudaStream_t s) {
    if (st.sp_inverse && st.sp_sums)
        return st.sp_off == 2
                   ? sums_dispatch<T, 2>(st, in, out, batch, adjoint, wide_in, wide_out, s)
                   : sums_dispatch<T, 1>(st, in, out, batch, adjoint, wide_in, wide_out, s);
    if (st.sp_inverse)
        return st.sp_off == 2 ? inverse_typed<T, 2>(st, in, out, batch, adjoint, s)
                              : inverse_typed<T, 1>(st, in, out, batch, adjoint, s);
    return st.sp_off == 2 ? forward_typed<T, 2>(st, in, out, batch, adjoint, s)
                          : forward_typed<T, 1>(st, in, out, batch, adjoint, s);
}

}  // namespace

namespace {

// ln W at the ends of [0, n) for factor f of F (see k_sum_tables), before normalisation.
void weight_range(const FactorSpec& F, int f, double* lo, double* hi) {
    const double par = F.par0 + F.dir * (double)f, s = par + F.b, last = (double)(F.n - 1);
    if (F.family == SP_ULTRA) {
        *lo = std::log(par);
        *hi = std::log(par + last);
        return;
    }
    auto lnw = [&](double j) {
        return std::log(2.0 * j + s + 1.0) + std::lgamma(j + s + 1.0) - std::lgamma(j + F.b + 1.0);
    };
    *lo = std::log((F.b + 1.0) / (s + 3.0)) + lnw(1.0);
    *hi = F.n > 1 ? lnw(last) : *lo;
}

bool sums_serve(const FactorSpec& F, int prec) {
    for (int f = 0; f < F.M && F.family != SP_ULTRA; ++f) {
        double lo, hi;
        weight_range(F, f, &lo, &hi);
        if (!(std::fabs(hi - lo) <= sum_range(prec))) return false;
    }
    return true;
}

template <typename A>
int sum_tables(Step& st, const FactorSpec& F, cudaStream_t s) {
    double* g = nullptr;  // Gamma ratios of one factor (Jacobi; entry 1 is read even for n = 1)
    const int64_t count = std::max<int64_t>(F.n, 2);
    if (F.family == SP_JACOBI) TDH_TRY(dev_alloc_t(&g, (size_t)count));
    int rc = TDH_OK;
    for (int f = 0; rc == TDH_OK && f < F.M; ++f) {
        double lo, hi;
        weight_range(F, f, &lo, &hi);
        const double par = F.par0 + F.dir * (double)f;
        if (g) rc = gamma_ratio_launch(par + F.b + 1.0, F.b + 1.0, count, g, s);
        if (rc != TDH_OK) break;
        const double scale = std::exp(-std::min(lo, hi));
        st.sp_gain[f] =
            F.family == SP_ULTRA ? 1.0f : (float)std::exp2(-std::ceil(std::fabs(hi - lo) / M_LN2));
        k_sum_tables<A><<<blocks_for(F.ld), kThreads, 0, s>>>(
            F, f, g, scale, st.scale_out, st.scale_in, static_cast<A*>(st.sp_tab));
        if (cudaGetLastError() != cudaSuccess) {
            set_error("back-substitution tables: launch failed");
            rc = TDH_ERR_CUDA;
        }
    }
    if (g) {
        cudaStreamSynchronize(s);
        dev_free(g);
    }
    return rc;
}

}  // namespace

int sparse_prepare(Step& st, int prec, cudaStream_t s) {
    if (st.sp_M < 1 || st.sp_M > kMaxM) {
        set_error("sparse-factor steps support 1..%d factors (got %d)", kMaxM, st.sp_M);
        return TDH_ERR_UNSUPPORTED;
    }
    if (st.sp_off != 1 && st.sp_off != 2) {
        set_error("sparse-factor band offset must be 1 or 2");
        return TDH_ERR_INVALID_ARG;
    }
    FactorSpec F{};
    F.family = st.sp_family;
    F.off = st.sp_off;
    F.M = st.sp_M;
    F.inverse = st.sp_inverse;
    F.flip = st.sp_flip;
    F.par0 = st.sp_par0;
    F.dir = st.sp_dir;
    F.b = st.sp_b;
    F.n = st.n;
    F.ld = (st.n + 2 + 3) / 4 * 4;  // float4 rows stay 16-byte aligned
    st.sp_ld = F.ld;
    if (!st.sp_inverse || !sums_serve(F, prec))
        st.sp_sums = 0;
    else if (st.sp_alone)
        st.sp_sums = 1;
    else
        st.sp_sums = prec != TDH_FP64 ? 2 : 0;
    const int rows = st.sp_inverse && !st.sp_sums ? kInvRows : 2;
    const size_t esz = prec != TDH_FP64 && st.sp_sums != 2 ? 4 : 8;
    TDH_TRY(dev_alloc(&st.sp_tab, esz * (size_t)F.ld * rows * st.sp_M));
    if (st.sp_sums == 2) return sum_tables<FF>(st, F, s);
    if (st.sp_sums)
        return prec != TDH_FP64 ? sum_tables<float>(st, F, s) : sum_tables<double>(st, F, s);
    const unsigned blocks = blocks_for(F.ld * F.M);
    if (prec != TDH_FP64)
        k_sparse_tables<float><<<blocks, kThreads, 0, s>>>(F, st.scale_out, st.scale_in,
                                                           static_cast<float*>(st.sp_tab));
    else
        k_sparse_tables<double><<<blocks, kThreads, 0, s>>>(F, st.scale_out, st.scale_in,
                                                            static_cast<double*>(st.sp_tab));
    TDH_CUDA(cudaGetLastError());
    return TDH_OK;
}

int sparse_check(const Step& st, int prec, int64_t batch, bool inplace) {
    static_assert(SumTile<float>::tile == Scan<float>::tile &&
                      SumTile<FF>::tile == Scan<float>::tile &&
                      SumTile<double>::tile == Scan<double>::tile,
                  "sums and affine scans take the same batches");
    if (!st.sp_inverse) {
        const bool whole = prec != TDH_FP64 && st.sp_M == 1 && st.n % 4 == 0 && !inplace;
        if (!whole && batch * ((st.n + kTile - 1) / kTile) > INT32_MAX) {
            set_error("sparse factors: batch * tiles above 2^31");
            return TDH_ERR_UNSUPPORTED;
        }
        return TDH_OK;
    }
    const int64_t tile = prec != TDH_FP64 ? Scan<float>::tile : Scan<double>::tile;
    if (batch * ((st.n + tile - 1) / tile) > INT32_MAX) {
        set_error("back-substitution: batch * tiles above 2^31");
        return TDH_ERR_UNSUPPORTED;
    }
    return TDH_OK;
}

int sparse_launch(const Step& st, int prec, const void* in, void* out, int64_t batch, int adjoint,
                  bool wide_in, bool wide_out, cudaStream_t s) {
    if (prec != TDH_FP64)
        return launch_typed<float>(st, in, out, batch, adjoint, wide_in, wide_out, s);
    return launch_typed<double>(st, in, out, batch, adjoint, wide_in, wide_out, s);
}

}  // namespace tdh
