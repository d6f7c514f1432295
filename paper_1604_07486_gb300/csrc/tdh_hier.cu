// Kernels and host side of the hierarchical T o H product (tdh_hier.cuh).
//
// Launches of a step: k_hier_up forms the moments of every box, k_hier_top (long vectors)
// exchanges those of the 2048-boxes, k_hier_far the smaller boxes' and passes the local
// expansions down, k_hier_near adds the near field and writes the result; each starts while the
// one before it drains (programmatic dependent launch).  Short vectors, few of them: one
// launch of k_hier_direct.  Vectors are independent; a CTA or warp takes a few of them, so every
// table entry it forms serves all of them.  n = 2^16 x 256 float32: 160 us (the FFT form: 2120;
// a copy of the batch: 20), n = 2^16 x 32 float64: 818 us (21760).
#include <algorithm>
#include <cmath>
#include <vector>

#include "tdh_hier.cuh"

namespace tdh {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTopKernel = 32;  // 2048-boxes from which their exchange is a kernel of its own
constexpr int kTopSplit = 8;  // ways the 2048-boxes' exchange is split over a CTA's threads

template <typename T>
struct HierParams {
    const T* in;
    T* out;
    int64_t n;       // coefficients per vector (dense)
    int64_t npk;     // NC * the padded length per channel (index reversal, table ends)
    int64_t batch;   // vectors of this launch
    int64_t bpad;    // vectors per box row of the moment arrays
    const T* s;
    const T* hh;
    const T* lw;     // leaf weights [P][32]
    const T* tr;     // transfer weights [3][4][P][P]
    const T* din;
    const T* dout;
    const T* a00;    // entry (0, 0) applied directly (null: in the tables)
    T* mom[kHierLevels];
    int leaf0, leaves;  // leaves [leaf0, leaves) hold coefficients (dense)
    int rev, sign_in, sign_out;
    int aligned;        // dense: every vector starts on a 16-byte boundary
    T* loc;             // leaf expansions [leaf][bpad][P][NC] (null: no far field)
    int nseg, seg_leaves, nvt, unvt;  // far segments; vectors per CTA (far, moments)
    T* top;             // 2048-boxes' exchange, [group][ntop][NC][nvt][P] (null: by k_hier_far)
    int ntop;           // 2048-boxes of a vector
    const T* st;        // s and h at the 2048-boxes' points (k_hier_top)
    const T* ht;
    int run;            // leaves a warp of the near kernel walks
    int64_t runs;       // such walks per vector group
    const int64_t* offs;  // ragged: vector i of the launch is list[i]
    const int* list;
    const int* count;     // vectors to convert, all launches of the call together
    int64_t first;        // index of the launch's first one among them
};

__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// 16 bytes of T
template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
    static constexpr int N = 4;
    float v[4];
    __device__ __forceinline__ void load(const float* p) {
        const float4 q = *reinterpret_cast<const float4*>(p);
        v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    }
    __device__ __forceinline__ void store(float* p) const {
        *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
    }
};
template <>
struct Vec16<double> {
    static constexpr int N = 2;
    double v[2];
    __device__ __forceinline__ void load(const double* p) {
        const double2 q = *reinterpret_cast<const double2*>(p);
        v[0] = q.x, v[1] = q.y;
    }
    __device__ __forceinline__ void store(double* p) const {
        *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
    }
};

// Where vector g of the launch starts and how long it is (length 0: none).
template <typename T, bool RAGGED>
__device__ __forceinline__ void vector_at(const HierParams<T>& P, int64_t g, int64_t* base,
                                          int64_t* len) {
    if constexpr (RAGGED) {
        if (g < P.batch && P.first + g < *P.count) {
            const int64_t v = P.list[g];
            *base = P.offs[v];
            *len = P.offs[v + 1] - *base;
            return;
        }
        *base = 0;
        *len = 0;
    } else {
        *base = g * P.n;
        *len = g < P.batch ? P.n : 0;
    }
}

// One past the last leaf any vector of the launch's vector group starting at g0 needs
// (ragged vectors are sorted, longest first).
template <typename T, int NC, bool RAGGED>
__device__ __forceinline__ int group_leaves(const HierParams<T>& P, int64_t g0) {
    if constexpr (!RAGGED) {
        return P.leaves;
    } else {
        int64_t base, len;
        vector_at<T, true>(P, g0, &base, &len);
        return (int)((len + NC * kHierLeaf - 1) / (NC * kHierLeaf));
    }
}

// Scaled input at packed position kp of a vector (0 outside it).
template <typename T>
__device__ __forceinline__ T scaled_input(const HierParams<T>& P, const T* x, int64_t len,
                                          int64_t kp) {
    const int64_t k = P.rev ? P.npk - 1 - kp : kp;
    if (k < 0 || k >= len) return T(0);
    const T v = x[k] * P.din[k];
    return (P.sign_in && (k & 1)) ? -v : v;
}

// Two values of T that go through the same operation: one 64-bit register operand in float32
// (fma.rn.f32x2: as many multiply-adds per cycle as scalar ones in half the instructions, which
// leaves issue slots to the loads), two scalar operations in float64.
using F2 = float2;
struct __align__(16) D2 {
    double x, y;
};
template <typename T>
struct PairOf;
template <>
struct PairOf<float> {
    using t = F2;
};
template <>
struct PairOf<double> {
    using t = D2;
};
__device__ __forceinline__ F2 pair_zero(float) { return make_float2(0.0f, 0.0f); }
__device__ __forceinline__ D2 pair_zero(double) { return D2{0.0, 0.0}; }
__device__ __forceinline__ void pair_fma(F2& c, F2 a, F2 b) {  // c += a b
    c = __ffma2_rn(a, b, c);
}
__device__ __forceinline__ void pair_fma(D2& c, D2 a, D2 b) {
    c.x = fma(a.x, b.x, c.x);
    c.y = fma(a.y, b.y, c.y);
}
__device__ __forceinline__ F2 pair_mul(F2 a, F2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ D2 pair_mul(D2 a, D2 b) { return D2{a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ F2 pair_make(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ D2 pair_make(double x, double y) { return D2{x, y}; }
__device__ __forceinline__ float pair_x(F2 a) { return a.x; }
__device__ __forceinline__ float pair_y(F2 a) { return a.y; }
__device__ __forceinline__ double pair_x(D2 a) { return a.x; }
__device__ __forceinline__ double pair_y(D2 a) { return a.y; }
// two consecutive pairs at p (16-byte aligned)
__device__ __forceinline__ void pair_load2(const F2* p, F2& a, F2& b) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void pair_load2(const D2* p, D2& a, D2& b) {
    const double2 q0 = *reinterpret_cast<const double2*>(p);
    const double2 q1 = *reinterpret_cast<const double2*>(p + 1);
    a = D2{q0.x, q0.y};
    b = D2{q1.x, q1.y};
}

__device__ __forceinline__ void load_pair(const float* p, float& a, float& b) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    a = q.x, b = q.y;
}
__device__ __forceinline__ void load_pair(const double* p, double& a, double& b) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    a = q.x, b = q.y;
}

// Coefficients k, k + 1 of a vector of len coefficients (0 outside it).
template <typename T>
__device__ __forceinline__ void load_two(const T* x, int64_t k, int64_t len, T& a, T& b) {
    if (k >= 0 && k + 1 < len && ((reinterpret_cast<uintptr_t>(x + k) & (2 * sizeof(T) - 1)) == 0)) {
        if constexpr (sizeof(T) == 4) {
            const float2 q = *reinterpret_cast<const float2*>(x + k);
            a = q.x, b = q.y;
        } else {
            const double2 q = *reinterpret_cast<const double2*>(x + k);
            a = q.x, b = q.y;
        }
    } else {
        a = (k >= 0 && k < len) ? x[k] : T(0);
        b = (k + 1 >= 0 && k + 1 < len) ? x[k + 1] : T(0);
    }
}
template <typename T>
__device__ __forceinline__ void store_two(T* y, int64_t k, int64_t len, T a, T b) {
    if (k >= 0 && k + 1 < len && ((reinterpret_cast<uintptr_t>(y + k) & (2 * sizeof(T) - 1)) == 0)) {
        if constexpr (sizeof(T) == 4)
            *reinterpret_cast<float2*>(y + k) = make_float2(a, b);
        else
            *reinterpret_cast<double2*>(y + k) = make_double2(a, b);
    } else {
        if (k >= 0 && k < len) y[k] = a;
        if (k + 1 >= 0 && k + 1 < len) y[k + 1] = b;
    }
}

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src)
                 : "memory");
}
// one value (4 or 8 bytes), or zero
template <int BYTES>
__device__ __forceinline__ void cp_async_small(void* dst, const void* src, bool valid) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(dst)),
                 "l"(src), "n"(BYTES), "r"(valid ? BYTES : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// ------------------------------------------------------------------------------- moments
//
// A CTA forms the moments of one 2048-box (64 leaves, their parents, ...) for unvt vectors.  A
// warp takes one leaf of VW vectors at a time: lane (p, v) holds the 32 weights L_p in
// registers, so each 16-byte shared load of inputs feeds 16 bytes' worth of multiply-adds; the
// next leaf's inputs are loaded meanwhile.  Bound by shared-memory reads (LSU 65 % busy, their
// latency the main stall): 41 us at n = 2^16 x 256 float32, whose inputs take 10 us to read; in
// float64 by the FP64 pipe (83 % busy): 131 us at 2^16 x 32.
template <typename T, int NC, bool RAGGED>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 4 : 2) k_hier_up(const __grid_constant__ HierParams<T> P) {
    constexpr int NP = HierP<T>::P;
    constexpr int VW = 32 / NP;
    constexpr int XW = NC * kHierLeaf;                 // inputs of a leaf
    constexpr int XS = XW + 16 / (int)sizeof(T);       // padded row
    constexpr int QV = Vec16<T>::N;
    constexpr int LPR = XW / 2;                        // lanes of a row (two inputs each)
    constexpr int RPI = 32 / LPR;                      // rows per load instruction
    constexpr int NL = VW / RPI > 0 ? VW / RPI : 1;    // load instructions per leaf
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // (ragged: the lists were written by the previous kernel, and no kernel after this one may
    // read them before they are there, so the next starts only from here on)
    if constexpr (RAGGED) pdl_wait();
    pdl_trigger();
    const int ntop = (P.leaves + kHierTopLeaves - 1) / kHierTopLeaves;
    const int top = blockIdx.x % ntop;
    const int64_t g0 = (int64_t)(blockIdx.x / ntop) * P.unvt;
    const int leaves = group_leaves<T, NC, RAGGED>(P, g0 / P.nvt * P.nvt);
    const int l0 = top * kHierTopLeaves;
    const int nl = min(kHierTopLeaves, leaves - l0);
    if (nl <= 0 || l0 + nl <= P.leaf0) return;
    const int nl4 = (nl + 3) & ~3;                     // whole sibling groups
    T* xw = reinterpret_cast<T*>(smem_raw) + warp * VW * XS;
    T* ms0 = reinterpret_cast<T*>(smem_raw) + kWarps * VW * XS;
    const int row = NC * P.unvt * NP;                  // one box's moments
    T* ms1 = ms0 + (size_t)kHierTopLeaves * row;
    T* ms2 = ms1 + (size_t)(kHierTopLeaves / 4) * row;
    T* tw = ms2 + (size_t)(kHierTopLeaves / 16) * row;  // transfer weights
    for (int i = tid; i < 12 * NP * NP; i += kThreads) tw[i] = P.tr[i];
    const int p = lane % NP, vq = lane / NP;
    T lw[kHierLeaf];
#pragma unroll
    for (int a = 0; a < kHierLeaf; ++a) lw[a] = P.lw[p * kHierLeaf + a];
    const int64_t boxrow = (int64_t)NC * P.bpad * NP;
    // row rv of load i is vector i RPI + lane / LPR; a lane loads two neighbouring inputs (in
    // reversed order they change places)
    const int rl = lane / LPR, col = 2 * (lane % LPR);
    const T* vx[NL];
    int64_t vlen[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i) {
        const int v = i * RPI + rl;
        int64_t base = 0, len = 0;
        if (v < VW) vector_at<T, RAGGED>(P, g0 + v, &base, &len);
        vx[i] = P.in + base;
        vlen[i] = len;
    }
    T xa[NL], xb[NL], da = T(0), db = T(0);
    auto load = [&](int leaf) {
        const int64_t kp = (int64_t)leaf * XW + col;
        const int64_t k = P.rev ? P.npk - 2 - kp : kp;
        load_two(P.din, k, P.n, da, db);
        if (P.sign_in) {
            if (k & 1)
                da = -da;
            else
                db = -db;
        }
        // whole leaf inside and two-value aligned: plain loads
        if (!RAGGED && P.aligned && k + 1 < P.n && k >= 0) {
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                xa[i] = xb[i] = T(0);
                if (vlen[i] > 0) load_pair(vx[i] + k, xa[i], xb[i]);
            }
        } else {
#pragma unroll
            for (int i = 0; i < NL; ++i) load_two(vx[i], k, vlen[i], xa[i], xb[i]);
        }
    };
    const int first = l0 + warp;
    if (first < l0 + nl) load(first);
    for (int li = warp; li < nl4; li += kWarps) {
        const int leaf = l0 + li;
        T acc[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = T(0);
        if (li < nl) {
            __syncwarp();
#pragma unroll
            for (int i = 0; i < NL; ++i) {
                const int v = i * RPI + rl;
                const T a = xa[i] * da, b = xb[i] * db;
                if (v < VW) {
                    xw[v * XS + col] = P.rev ? b : a;
                    xw[v * XS + col + 1] = P.rev ? a : b;
                }
            }
            __syncwarp();
            if (li + kWarps < nl) load(leaf + kWarps);
            const T* xv = xw + vq * XS;
#pragma unroll
            for (int i = 0; i < XW; i += QV) {
                Vec16<T> q;
                q.load(xv + i);
#pragma unroll
                for (int j = 0; j < QV; ++j) acc[(i + j) % NC] += lw[(i + j) / NC] * q.v[j];
            }
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            ms0[(size_t)li * row + (c * P.unvt + vq) * NP + p] = acc[c];
            if (li < nl)
                P.mom[0][leaf * boxrow + ((int64_t)c * P.bpad + g0 + vq) * NP + p] = acc[c];
        }
    }
    // parents from children, level by level: a thread takes HPT of one box's points for one
    // vector, their weights the same for all vectors and channels
    int nb = nl4 / 4;
    const T* src = ms0;
    T* dst = ms1;
    constexpr int HPT = sizeof(T) == 4 ? NP / 2 : 2, SPL = NP / HPT;
    for (int l = 1; l < kHierLevels; ++l) {
        __syncthreads();
        const int nbp = l < kHierLevels - 1 ? (nb + 3) & ~3 : nb;
        const int cvs = NC * P.unvt;
        for (int i = tid; i < nbp * SPL * cvs; i += kThreads) {
            const int cv = i % cvs, hb = i / cvs;
            const int box = hb / SPL, p0 = hb % SPL * HPT;
            T acc[HPT];
#pragma unroll
            for (int pp = 0; pp < HPT; ++pp) acc[pp] = T(0);
            if (box < nb) {
#pragma unroll 1
                for (int c = 0; c < 4; ++c) {
                    const T* m = src + (size_t)(4 * box + c) * row + cv * NP;
                    const T* w = tw + (((l - 1) * 4 + c) * NP + p0) * NP;
#pragma unroll
                    for (int q = 0; q < NP; q += QV) {
                        Vec16<T> mv;
                        mv.load(m + q);
#pragma unroll
                        for (int pp = 0; pp < HPT; ++pp) {
                            Vec16<T> wv;
                            wv.load(w + pp * NP + q);
#pragma unroll
                            for (int j = 0; j < QV; ++j) acc[pp] += wv.v[j] * mv.v[j];
                        }
                    }
                }
                const int64_t gb = (l0 >> (2 * l)) + box;
                const int c = cv / P.unvt, v = cv % P.unvt;
                T* o = P.mom[l] + gb * boxrow + ((int64_t)c * P.bpad + g0 + v) * NP + p0;
#pragma unroll
                for (int pp = 0; pp < HPT; ++pp) o[pp] = acc[pp];
            }
            if (l < kHierLevels - 1) {
                T* o = dst + (size_t)box * row + cv * NP + p0;
#pragma unroll
                for (int pp = 0; pp < HPT; ++pp) o[pp] = acc[pp];
            }
        }
        src = dst;
        dst = ms2;
        nb = nbp / 4;
    }
}

// ------------------------------------------------------------------------------ far field
//
// A CTA forms the local expansions of one segment's leaves (seg_leaves leaves: 16 or 4) for NVT
// vectors: the exchange of the segment's boxes of every level (and of the boxes above it, on
// its path), then parents into children; the leaves' expansions go to P.loc
// ([leaf][vector][P][NC], channels in their natural order).
//
// Exchange: a warp takes one box, its lanes the box's points, channels and VTL groups of VPT
// vectors, so a coefficient s h that a lane forms (table offsets of the points are constants of
// the level) serves VPT vectors.  Children: a thread takes one box of one vector whole, its
// weights broadcast from shared memory.  Bound by shared-memory reads (LSU 65 % busy) and the
// barriers between its phases: 52 us at n = 2^16 x 256 float32; in float64 by the FP64 pipe (76 %
// busy): 364 us at 2^16 x 32.
template <typename T, int NC, int NVT>
struct FarShape {
    static constexpr int NP = HierP<T>::P;
    static constexpr int VTL = 32 / (NP * NC) < NVT ? 32 / (NP * NC) : NVT;  // vector groups
    static constexpr int VPT = NVT / VTL;
    static constexpr int erow = NC * NVT * NP;  // one box's expansions
    static constexpr int trw = 3 * 4 * NP * NP;
    static constexpr int MG = VPT * NP + 16 / (int)sizeof(T);  // staged moments of a lane group
};

// One box of level L (index i): the far boxes' moments at this lane's point.
template <typename T, int NC, int VPT, int L>
__device__ __forceinline__ void far_box(const T* sp, const T* hp, const T* m0, int64_t boxrow,
                                        int d0, int d1, int step, T (&acc)[VPT]) {
    constexpr int NP = HierP<T>::P;
    constexpr int QV = Vec16<T>::N;
    constexpr int size = hier_size(L);
    const T* m = m0 + d0 * boxrow;
    sp += d0 * size;
    hp += d0 * size;
#pragma unroll 1
    for (int d = d0; d < d1; d += step) {
#pragma unroll
        for (int q0 = 0; q0 < NP; q0 += QV) {
            T cf[QV];
#pragma unroll
            for (int j = 0; j < QV; ++j)
                cf[j] = sp[hier_point<NP>(L, q0 + j)] * hp[hier_point<NP>(L, q0 + j)];
#pragma unroll
            for (int u = 0; u < VPT; ++u) {
                Vec16<T> mv;
                mv.load(m + u * NP + q0);
#pragma unroll
                for (int j = 0; j < QV; ++j) acc[u] += cf[j] * mv.v[j];
            }
        }
        m += step * boxrow;
        sp += step * size;
        hp += step * size;
    }
}

// Long vectors: the exchange of the 2048-boxes, one CTA per box and NVT vectors, the far boxes
// split over its warps; to P.top ([group][box][NC][NVT][P]).  (Within k_hier_far every segment
// of a 2048-box would repeat it: fine for a few boxes, 3/4 of that kernel at 512 of them.)  The
// points lie a sector or more apart in s and h, so the factors are read from tables of their
// own (16 lanes' rows contiguous): 105 -> 44 us at n = 2^20 x 16 float32.
template <typename T, int NC, int NVT, bool RAGGED>
__global__ void __launch_bounds__(kThreads) k_hier_top(const __grid_constant__ HierParams<T> P) {
    using F = FarShape<T, NC, NVT>;
    constexpr int NP = F::NP, VTL = F::VTL, VPT = F::VPT, erow = F::erow;
    constexpr int TOP = kHierLevels - 1;
    __shared__ T part[kWarps * erow];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_trigger();
    const int i = blockIdx.x % P.ntop;
    const int64_t grp = blockIdx.x / P.ntop, g0 = grp * NVT;
    pdl_wait();  // the moments were written by the previous kernel
    const int leaves = group_leaves<T, NC, RAGGED>(P, g0);
    const int nb = (leaves + kHierTopLeaves - 1) / kHierTopLeaves;
    if (i >= nb) return;
    const int64_t boxrow = (int64_t)NC * P.bpad * NP;
    const int p = lane % NP, vt = (lane / NP) % VTL, c = lane / (NP * VTL);
    if (c < NC) {
        using P2 = typename PairOf<T>::t;
        const T* st = P.st + p * NP;
        const T* ht = P.ht + (((int64_t)2 * i * NC + c) * NP + p) * NP;
        const T* m = P.mom[TOP] + i * boxrow + ((int64_t)c * P.bpad + g0 + vt * VPT) * NP;
        P2 acc[VPT];  // sums over the even and the odd points
#pragma unroll
        for (int u = 0; u < VPT; ++u) acc[u] = pair_zero(T(0));
#pragma unroll 1
        for (int64_t d = 2 + warp; d < nb - i; d += kWarps) {
#pragma unroll
            for (int q = 0; q < NP; q += 4) {
                P2 s0, s1, h0, h1;
                pair_load2(reinterpret_cast<const P2*>(st + d * (NP * NP) + q), s0, s1);
                pair_load2(reinterpret_cast<const P2*>(ht + d * (NC * NP * NP) + q), h0, h1);
                s0 = pair_mul(s0, h0);
                s1 = pair_mul(s1, h1);
#pragma unroll
                for (int u = 0; u < VPT; ++u) {
                    P2 y0, y1;
                    pair_load2(reinterpret_cast<const P2*>(m + d * boxrow + u * NP + q), y0, y1);
                    pair_fma(acc[u], s0, y0);
                    pair_fma(acc[u], s1, y1);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < VPT; ++u)
            part[warp * erow + (c * NVT + vt * VPT + u) * NP + p] = pair_x(acc[u]) + pair_y(acc[u]);
    }
    __syncthreads();
    for (int e = tid; e < erow; e += kThreads) {
        T a = part[e];
#pragma unroll
        for (int w = 1; w < kWarps; ++w) a += part[w * erow + e];
        P.top[(grp * P.ntop + i) * erow + e] = a;
    }
}

template <typename T, int NC, int NVT, bool RAGGED>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 ? 3 : 2) k_hier_far(
    const __grid_constant__ HierParams<T> P) {
    using F = FarShape<T, NC, NVT>;
    constexpr int NP = F::NP, VTL = F::VTL, VPT = F::VPT, erow = F::erow;
    constexpr int QV = Vec16<T>::N;
    constexpr int TOP = kHierLevels - 1;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int xn[kHierLevels][NP];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_trigger();
    const int nseg = P.nseg, SL = P.seg_leaves;
    const int seg = blockIdx.x % nseg;
    const int64_t g0 = (int64_t)(blockIdx.x / nseg) * NVT;
    const int leaves = group_leaves<T, NC, RAGGED>(P, g0);
    const int l0 = seg * SL;
    if (l0 >= leaves || l0 + SL <= P.leaf0) {
        pdl_wait();  // the launch must not complete before the moments' does
        return;
    }
    const int a0 = l0 * kHierLeaf;
    // shared memory: s window [-32, 256), h window, transfer weights, expansions
    T* sw = reinterpret_cast<T*>(smem_raw) + kHierSZero;
    constexpr int SW = 8 * kHierLeaf;
    T* hw = sw + SW;
    const int HW = 2 * SL * kHierLeaf + 10 * kHierLeaf;
    T* tw = hw + HW;
    const int n1 = max(1, SL / 4), n2 = max(1, SL / 16);
    // leaves' moments [box][channel][NVT][P], rows of a box padded so that the lanes' vector
    // groups and channels meet other banks
    constexpr int MG = F::MG, MC = VTL * MG;   // a lane group's vectors, one channel's row
    T* mw = tw + F::trw;
    T* e3 = mw + (SL + 7) * NC * MC;            // [kTopSplit] parts of the 2048-box's
    T* e2 = e3 + kTopSplit * erow;
    T* e1 = e2 + n2 * erow;
    T* e0 = e1 + n1 * erow;
    for (int i = tid; i < SW + kHierSZero; i += kThreads) sw[i - kHierSZero] = P.s[i - kHierSZero];
    for (int i = tid; i < HW; i += kThreads) {
        const int64_t g = 2 * (int64_t)a0 + i;
        hw[i] = g < 2 * (P.npk / NC) + kHierHPad - 1 ? P.hh[g] : T(0);
    }
    for (int i = tid; i < F::trw; i += kThreads) tw[i] = P.tr[i];
    if (tid == 0)
#pragma unroll
        for (int i = 0; i < kHierLevels * NP; ++i) xn[i / NP][i % NP] = hier_point<NP>(i / NP, i % NP);
    __syncthreads();
    pdl_wait();  // the moments were written by the previous kernel
    // ---- exchange: leaves, their parents, ..., the parts of the 2048-box
    const int64_t boxrow = (int64_t)NC * P.bpad * NP;
    {
        constexpr int CPC = NVT * NP / QV;      // 16-byte chunks of a channel's row
        const int nbox = min(SL + 7, leaves - l0);
        for (int i = tid; i < nbox * NC * CPC; i += kThreads) {
            const int q = i % CPC, bc = i / CPC;
            constexpr int CPG = VPT * NP / QV;  // chunks of a lane group
            cp_async16(mw + bc * MC + q / CPG * MG + q % CPG * QV,
                       P.mom[0] + (l0 + bc / NC) * boxrow +
                           ((int64_t)(bc % NC) * P.bpad + g0) * NP + q * QV);
        }
        cp_async_wait_all();
        __syncthreads();
    }
    const int p = lane % NP, vt = (lane / NP) % VTL, c = lane / (NP * VTL);
    const int nbx = SL + n1 + n2 + (P.top ? 0 : kTopSplit);
    for (int bx = warp; bx < nbx && c < NC; bx += kWarps) {
        T acc[VPT];
#pragma unroll
        for (int u = 0; u < VPT; ++u) acc[u] = T(0);
        const int64_t mo = ((int64_t)c * P.bpad + g0 + vt * VPT) * NP;
        T* e;
        if (bx < SL) {
            const int i = l0 + bx;
            far_box<T, NC, VPT, 0>(sw - xn[0][p], hw + 2 * bx * kHierLeaf + xn[0][p] + c,
                                   mw + (bx * NC + c) * MC + vt * MG, NC * MC, 2,
                                   min(8 - (i & 3), leaves - i), 1, acc);
            e = e0 + bx * erow;
        } else if (bx < SL + n1) {
            const int i = (l0 >> 2) + bx - SL, nb = (leaves + 3) >> 2;
            far_box<T, NC, VPT, 1>(P.s - xn[1][p], P.hh + (int64_t)2 * i * hier_size(1) + xn[1][p] + c,
                                   P.mom[1] + i * boxrow + mo, boxrow, 2,
                                   min(8 - (i & 3), nb - i), 1, acc);
            e = e1 + (bx - SL) * erow;
        } else if (bx < SL + n1 + n2) {
            const int i = (l0 >> 4) + bx - SL - n1, nb = (leaves + 15) >> 4;
            far_box<T, NC, VPT, 2>(P.s - xn[2][p], P.hh + (int64_t)2 * i * hier_size(2) + xn[2][p] + c,
                                   P.mom[2] + i * boxrow + mo, boxrow, 2,
                                   min(8 - (i & 3), nb - i), 1, acc);
            e = e2 + (bx - SL - n1) * erow;
        } else {
            const int i = l0 >> 6, nb = (leaves + 63) >> 6, part = bx - SL - n1 - n2;
            far_box<T, NC, VPT, 3>(P.s - xn[3][p], P.hh + (int64_t)2 * i * hier_size(3) + xn[3][p] + c,
                                   P.mom[3] + i * boxrow + mo, boxrow, 2 + part, nb - i, kTopSplit,
                                   acc);
            e = e3 + part * erow;
        }
        e += (c * NVT + vt * VPT) * NP + p;
#pragma unroll
        for (int u = 0; u < VPT; ++u) e[u * NP] = acc[u];
    }
    __syncthreads();
    for (int i = tid; i < erow; i += kThreads) {
        T a;
        if (P.top) {
            a = P.top[(g0 / NVT * P.ntop + (l0 >> 6)) * erow + i];
        } else {
            a = e3[i];
#pragma unroll
            for (int k = 1; k < kTopSplit; ++k) a += e3[k * erow + i];
        }
        e3[i] = a;
    }
    // ---- parents into children; the leaves' expansions go out
#pragma unroll 1
    for (int l = TOP - 1; l >= 0; --l) {
        __syncthreads();
        const T* from = l == 2 ? e3 : l == 1 ? e2 : e1;
        T* to = l == 2 ? e2 : l == 1 ? e1 : e0;
        const int nb = l == 2 ? n2 : l == 1 ? n1 : SL, np = l == 2 ? 1 : l == 1 ? n2 : n1;
        for (int it = tid; it < nb * NC * NVT; it += kThreads) {
            const int v = it % NVT, cc = (it / NVT) % NC, bl = it / (NVT * NC);
            const int i = (l0 >> (2 * l)) + bl;
            const T* par = from + (np > 1 ? bl / 4 : 0) * erow + (cc * NVT + v) * NP;
            T* ch = to + bl * erow + (cc * NVT + v) * NP;
            const T* w = tw + (l * 4 + (i & 3)) * NP * NP;
            T out[NP], x[NP];
#pragma unroll
            for (int q = 0; q < NP; q += QV) {
                Vec16<T> o, f;
                o.load(ch + q);
                f.load(par + q);
#pragma unroll
                for (int j = 0; j < QV; ++j) {
                    out[q + j] = o.v[j];
                    x[q + j] = f.v[j];
                }
            }
#pragma unroll
            for (int pp = 0; pp < NP; ++pp) {
#pragma unroll
                for (int q = 0; q < NP; q += QV) {
                    Vec16<T> o;
                    o.load(w + pp * NP + q);
#pragma unroll
                    for (int j = 0; j < QV; ++j) out[q + j] += o.v[j] * x[pp];
                }
            }
#pragma unroll
            for (int q = 0; q < NP; q += QV) {
                Vec16<T> o;
#pragma unroll
                for (int j = 0; j < QV; ++j) o.v[j] = out[q + j];
                o.store(ch + q);
            }
        }
    }
    __syncthreads();
    {
        // out in whole 16-byte pieces: [leaf][vector][P][NC]
        constexpr int PPV = NC * NP / QV;       // pieces of a vector
        const int pieces = min(SL, leaves - l0) * NVT * PPV;
        for (int it = tid; it < pieces; it += kThreads) {
            const int w = it % PPV, v = (it / PPV) % NVT, bl = it / (PPV * NVT);
            Vec16<T> o;
#pragma unroll
            for (int j = 0; j < QV; ++j) {
                const int e = w * QV + j, q = e / NC, cc = P.rev ? NC - 1 - e % NC : e % NC;
                o.v[j] = e0[bl * erow + (cc * NVT + v) * NP + q];
            }
            o.store(P.loc + ((int64_t)(l0 + bl) * P.bpad + g0 + v) * (NC * NP) + w * QV);
        }
    }
}

// ----------------------------------------------------------------------------- near field
//
// A warp walks `run` leaves of NV vectors: leaf j's scaled inputs come into its own shared
// memory, give the off-diagonal block of leaf j - 1's rows, which are then complete (local
// expansion, output scaling, store), and the triangle of leaf j's.  No barrier between warps.
//
// The two half-warps take half of the vectors each, a lane rows r and r + 16.  Values are taken
// in pairs (two parities of one packed index, or two neighbouring indices), so one 16-byte
// broadcast of inputs feeds four pair operations per row pair, and the entries s h a lane forms
// serve all of its vectors.  n = 2^16 x 256 float32: 76 us, the FP32 pipe 48 % busy and the LSU
// 64 % (fused with the far field the whole product took 291 us against 160); two warps a
// scheduler leave the latency of the shared loads exposed, but four of half as many
// vectors load more and take 15 % longer.  n = 2^16 x 32 float64: 339 us, bound by the FP64 pipe.
template <typename T, int NC, int NV>
struct NearShape {
    static constexpr int NP = HierP<T>::P;
    static constexpr int NPR = NC * kHierLeaf / 2;             // pairs of a leaf
    static constexpr int CH = 16 / (int)sizeof(T);             // coefficients of a 16-byte chunk
    static constexpr int CPR = 2 * NPR / CH;                   // chunks of a leaf's row
    static constexpr int XS = NPR + (sizeof(T) == 4 ? 2 : 1);  // row stride, in pairs
    static constexpr int LS = NC * NP / 2;                     // pairs of an expansion, per vector
    static constexpr int HP = 3 * kHierLeaf;                   // Hankel window per step, in pairs
    static constexpr int LW = (NC == 2 ? NP : NP / 2) * kHierLeaf;
    // one CTA per SM
    static constexpr int warps = NV * (int)sizeof(T) >= 128 ? 8 : 16;
    // pairs of shared memory: of a warp (two input buffers), and of the CTA's tables (s pairs,
    // leaf weights)
    static constexpr int warp_pairs(bool ragged) {
        return 2 * NV * XS + HP + NV * LS + (ragged ? NV * 16 / (int)(2 * sizeof(T)) : 0);
    }
    static constexpr int table_pairs = 3 * kHierLeaf + LW;
};

template <typename T, int NC, int NV, bool REV, bool RAGGED>
__global__ void __launch_bounds__(32 * NearShape<T, NC, NV>::warps, 1) k_hier_near(
    const __grid_constant__ HierParams<T> P) {
    using S = NearShape<T, NC, NV>;
    using P2 = typename PairOf<T>::t;
    constexpr int KV = NV / 2;                       // vectors per half-warp
    constexpr int NPR = S::NPR, XS = S::XS, LS = S::LS, HP = S::HP, LW = S::LW;
    constexpr int CS = NC == 2 ? 1 : 2;              // packed indices per pair
    constexpr int CH = S::CH, CPR = S::CPR, RPI = 32 / CPR;
    constexpr int NIT = NV > RPI ? NV / RPI : 1;     // chunks per lane and leaf
    constexpr int NTH = 32 * S::warps;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    P2* sp = reinterpret_cast<P2*>(smem_raw) + kHierLeaf;  // s pairs [-32, 64)
    P2* lw = sp + 2 * kHierLeaf;                           // leaf weights [.][32]
    P2* xs = lw + LW + (size_t)warp * S::warp_pairs(RAGGED);
    P2* hp = xs + 2 * NV * XS;
    P2* lc = hp + HP;
    longlong2* vt = reinterpret_cast<longlong2*>(lc + NV * LS);  // ragged: {start, length}
    for (int i = tid; i < 3 * kHierLeaf; i += NTH) {
        const int m = i - kHierLeaf;
        const T s0 = P.s[m], s1 = P.s[m + 1];
        sp[m] = NC == 2 ? pair_make(s0, s0) : (REV ? pair_make(s1, s0) : pair_make(s0, s1));
    }
    for (int i = tid; i < LW; i += NTH) {
        const int q = i / kHierLeaf, a = i % kHierLeaf;
        lw[i] = NC == 2 ? pair_make(P.lw[i], P.lw[i])
                        : pair_make(P.lw[2 * q * kHierLeaf + a], P.lw[(2 * q + 1) * kHierLeaf + a]);
    }
    __syncthreads();
    const int64_t task = (int64_t)blockIdx.x * S::warps + warp;
    const int64_t g0 = task / P.runs * NV;
    const int i0 = P.leaf0 + (int)(task % P.runs) * P.run;
    bool far = false;
    int leaves = 0;
    if (g0 < P.batch) {
        leaves = group_leaves<T, NC, RAGGED>(P, g0);
        // a group's far field was formed with the leaves of the far kernel's group
        far = P.loc && group_leaves<T, NC, RAGGED>(P, g0 / P.nvt * P.nvt) > 2;
    }
    const int i1 = min(i0 + P.run, leaves);
    if (i0 >= i1) {
        pdl_wait();  // the launch must not complete before the previous one does
        return;
    }
    if constexpr (RAGGED) {
        for (int v = lane; v < NV; v += 32) {
            int64_t base, len;
            vector_at<T, true>(P, g0 + v, &base, &len);
            vt[v] = make_longlong2(base, len);
        }
        __syncwarp();
    }
    auto vec = [&](int v, int64_t* base, int64_t* len) {
        if constexpr (RAGGED) {
            const longlong2 q = vt[v];
            *base = q.x;
            *len = q.y;
        } else {
            vector_at<T, false>(P, g0 + v, base, len);
        }
    };
    // half-warp h takes vectors 2 k + h: neighbouring rows, whose broadcasts meet other banks
    const int half = lane >> 4, r = lane & 15;
    const int hmax = (int)(2 * (P.npk / NC)) + kHierHPad - 2;
    const int col = lane % CPR, rv = lane / CPR;  // a lane's chunk column and first row
    const int nv = RAGGED ? NV : (int)min((int64_t)NV, P.batch - g0);
    // natural index of a lane's chunk of leaf j
    auto chunk_at = [&](int j) -> int64_t {
        return (REV ? P.npk - (int64_t)(j + 1) * 2 * NPR : (int64_t)j * 2 * NPR) + col * CH;
    };
    // start the copy of leaf j's inputs (unscaled) into its buffer
    auto fetch = [&](int j) {
        const int64_t k = chunk_at(j);
        P2* xb = xs + (j & 1) * NV * XS;
        if (!RAGGED && P.aligned && k >= 0 && k + CH <= P.n) {
            const T* x = P.in + (g0 + rv) * P.n + k;
            T* to = reinterpret_cast<T*>(xb + rv * XS) + col * CH;
#pragma unroll
            for (int i = 0; i < NIT; ++i) {
                if (i * RPI + rv < nv) cp_async16(to, x);
                x += RPI * P.n;
                to += RPI * 2 * XS;
            }
        } else {
#pragma unroll 1
            for (int v = rv; v < NV; v += RPI) {
                int64_t base, len;
                vec(v, &base, &len);
                const T* x = P.in + base + k;
                T* to = reinterpret_cast<T*>(xb + v * XS) + col * CH;
                if (k >= 0 && k + CH <= len && (reinterpret_cast<uintptr_t>(x) & 15) == 0) {
                    cp_async16(to, x);
                } else {
#pragma unroll
                    for (int u = 0; u < CH; ++u) {
                        const bool in = k + u >= 0 && k + u < len;
                        cp_async_small<(int)sizeof(T)>(to + u, in ? x + u : P.in, in);
                    }
                }
            }
        }
    };
    // a lane's input scaling of leaf j, and its entries of leaf j's Hankel window (from 64 j - 32)
    T d[CH], hl[HP / 32], hh[HP / 32];
    auto tables = [&](int j) {
        const int64_t k = chunk_at(j);
#pragma unroll
        for (int u = 0; u < CH; ++u) {
            const int64_t kk = k + u;
            d[u] = kk >= 0 && kk < P.n ? P.din[kk] : T(0);
            if (P.sign_in && (kk & 1)) d[u] = -d[u];
        }
        const int hb = 2 * j * kHierLeaf - kHierLeaf + lane;
#pragma unroll
        for (int i = 0; i < HP / 32; ++i) {
            const int g = hb + 32 * i;
            hl[i] = g >= 0 && g < hmax ? P.hh[g] : T(0);
            hh[i] = g >= -1 && g < hmax ? P.hh[g + 1] : T(0);
        }
    };
    const P2* xv = xs;
    // primed pair q is natural pair q, or NPR - 1 - q when reversed
    auto two = [&](int k, int q, P2& x0, P2& x1) {
        if constexpr (REV)
            pair_load2(xv + 2 * k * XS + NPR - 2 - q, x1, x0);
        else
            pair_load2(xv + 2 * k * XS + q, x0, x1);
    };
    P2 acc[KV][2];
    // acc += entries of columns CS q ... (pairs q0 <= q < NPR) for rows r and r + 16
    auto both_rows = [&](const P2* s0, const P2* h0, int q0) {
#pragma unroll 1
        for (int q = q0; q < NPR; q += 2) {
            const int b = CS * q;
            const P2 a00 = pair_mul(s0[b], h0[b]);
            const P2 a01 = pair_mul(s0[b + CS], h0[b + CS]);
            const P2 a10 = pair_mul(s0[b - 16], h0[b + 16]);
            const P2 a11 = pair_mul(s0[b + CS - 16], h0[b + CS + 16]);
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                P2 x0, x1;
                two(k, q, x0, x1);
                pair_fma(acc[k][0], a00, x0);
                pair_fma(acc[k][1], a10, x0);
                pair_fma(acc[k][0], a01, x1);
                pair_fma(acc[k][1], a11, x1);
            }
        }
    };
    fetch(i0);
    cp_async_commit();
    tables(i0);
#pragma unroll 1
    for (int j = i0; j <= i1; ++j) {
        // ---- leaf j's inputs are here: scale what this lane copied
        cp_async_wait<0>();
        if (j < leaves) {
            T* to = reinterpret_cast<T*>(xs + (j & 1) * NV * XS + rv * XS) + col * CH;
#pragma unroll
            for (int i = 0; i < NIT; ++i) {
                if (i * RPI + rv < NV) {
                    Vec16<T> q;
                    q.load(to);
#pragma unroll
                    for (int u = 0; u < CH; ++u) q.v[u] *= d[u];
                    q.store(to);
                }
                to += RPI * 2 * XS;
            }
#pragma unroll
            for (int i = 0; i < HP / 32; ++i)
                hp[32 * i + lane] = REV ? pair_make(hh[i], hl[i]) : pair_make(hl[i], hh[i]);
        }
        __syncwarp();
        // ---- start what comes next: leaf j - 1's expansions and scaling, leaf j + 1's inputs
        T da[2], db[2];
        if (j > i0) {
            if (j == i0 + 1) pdl_wait();  // the expansions were written by the previous kernel
            if (far) {
                const T* e = P.loc + ((int64_t)(j - 1) * P.bpad + g0) * (NC * S::NP);
#pragma unroll
                for (int i = lane; i < NV * NC * S::NP / CH; i += 32)
                    cp_async16(reinterpret_cast<T*>(lc) + i * CH, e + i * CH);
            }
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                const int64_t kp = (int64_t)NC * ((int64_t)(j - 1) * kHierLeaf + r + 16 * rr);
                const int64_t k0 = REV ? P.npk - NC - kp : kp;
                da[rr] = db[rr] = T(0);
                if constexpr (NC == 2)
                    load_two(P.dout, k0, P.n, da[rr], db[rr]);
                else if (k0 >= 0 && k0 < P.n)
                    da[rr] = P.dout[k0];
                if (P.sign_out) {
                    if (k0 & 1)
                        da[rr] = -da[rr];
                    else
                        db[rr] = -db[rr];
                }
            }
        }
        cp_async_commit();
        if (j < i1 && j + 1 < leaves) {
            fetch(j + 1);
            tables(j + 1);
        }
        cp_async_commit();
        xv = xs + (j & 1) * NV * XS + half * XS;
        if (j > i0) {
            // ---- off-diagonal block, rows of leaf j - 1 and columns of leaf j:
            // l = 32 (j-1) + r + 32 j + b, window from 64 j - 32
            if (j < leaves) both_rows(sp + kHierLeaf - r, hp + r, 0);
            // ---- rows of leaf j - 1 are complete but for the far field
            if (far) {
                cp_async_wait<1>();
                __syncwarp();
#pragma unroll 1
                for (int q = 0; q < LS; q += 2) {
                    const P2 w00 = lw[q * kHierLeaf + r], w10 = lw[q * kHierLeaf + r + 16];
                    const P2 w01 = lw[(q + 1) * kHierLeaf + r];
                    const P2 w11 = lw[(q + 1) * kHierLeaf + r + 16];
#pragma unroll
                    for (int k = 0; k < KV; ++k) {
                        P2 x0, x1;
                        pair_load2(lc + (2 * k + half) * LS + q, x0, x1);
                        pair_fma(acc[k][0], w00, x0);
                        pair_fma(acc[k][1], w10, x0);
                        pair_fma(acc[k][0], w01, x1);
                        pair_fma(acc[k][1], w11, x1);
                    }
                }
            }
#pragma unroll
            for (int rr = 0; rr < 2; ++rr) {
                const int64_t kp = (int64_t)NC * ((int64_t)(j - 1) * kHierLeaf + r + 16 * rr);
                const int64_t k0 = REV ? P.npk - NC - kp : kp;
                const bool direct = k0 == 0 && P.a00;
                if (!RAGGED && P.aligned && !direct && k0 >= 0 && k0 + NC <= P.n) {
                    T* o = P.out + (g0 + half) * P.n + k0;
#pragma unroll
                    for (int k = 0; k < KV; ++k) {
                        if (2 * k + half < nv) {
                            if constexpr (NC == 2)
                                *reinterpret_cast<P2*>(o) =
                                    pair_mul(acc[k][rr], pair_make(da[rr], db[rr]));
                            else
                                *o = (pair_x(acc[k][rr]) + pair_y(acc[k][rr])) * da[rr];
                        }
                        o += 2 * P.n;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < KV; ++k) {
                        int64_t base, len;
                        vec(2 * k + half, &base, &len);
                        T* o = P.out + base;
                        T ya, yb = T(0);
                        if constexpr (NC == 2) {
                            ya = pair_x(acc[k][rr]) * da[rr];
                            yb = pair_y(acc[k][rr]) * db[rr];
                        } else {
                            ya = (pair_x(acc[k][rr]) + pair_y(acc[k][rr])) * da[rr];
                        }
                        if (direct && len > 0) ya += P.a00[0] * P.in[base];
                        if constexpr (NC == 2)
                            store_two(o, k0, len, ya, yb);
                        else if (k0 >= 0 && k0 < len)
                            o[k0] = ya;
                    }
                }
            }
        }
        if (j < i1) {
            // ---- triangle of leaf j: l = 64 j + r + b (s is zero left of the diagonal; rows
            // r + 16 meet no column below 16)
#pragma unroll
            for (int k = 0; k < KV; ++k) acc[k][0] = acc[k][1] = pair_zero(T(0));
            const P2* s0 = sp - r;
            const P2* h0 = hp + kHierLeaf + r;
#pragma unroll 1
            for (int q = 0; q < NPR / 2; q += 2) {
                const int b = CS * q;
                const P2 a00 = pair_mul(s0[b], h0[b]);
                const P2 a01 = pair_mul(s0[b + CS], h0[b + CS]);
#pragma unroll
                for (int k = 0; k < KV; ++k) {
                    P2 x0, x1;
                    two(k, q, x0, x1);
                    pair_fma(acc[k][0], a00, x0);
                    pair_fma(acc[k][0], a01, x1);
                }
            }
            both_rows(s0, h0, NPR / 2);
        }
        __syncwarp();  // every lane is done with the buffers this step read
    }
}

// --------------------------------------------------------------------------- direct product
//
// Short vectors, few of them: every entry of the triangle once, no far field (one launch).  A
// CTA stages the scaled inputs and the tables in shared memory; a warp takes one packed row
// of V vectors, lanes along the columns (s from the diagonal on, h and the inputs all read with
// consecutive lanes on consecutive places); where the rows are few, WR warps share one.  Bound by
// its launch in float32 (2.6 to 6 us), by the FP64 pipe in float64.
template <typename T, int NC, int V, int WR>  // WR warps share a row
__global__ void __launch_bounds__(kThreads) k_hier_direct(const __grid_constant__ HierParams<T> P,
                                                          int m) {
    constexpr int rows = kWarps / WR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nrow = (m + rows - 1) / rows;
    const int a0 = (int)(blockIdx.x % nrow) * rows;
    const int64_t g0 = (int64_t)(blockIdx.x / nrow) * V;
    const int w = m - a0;                       // columns a0 .. m - 1
    const int64_t k0 = P.rev ? P.npk - (int64_t)NC * m : 0;  // packed position of row 0
    const int64_t l0 = 2 * (k0 / NC + a0);      // Hankel index of (a0, a0)
    T* sm = reinterpret_cast<T*>(smem_raw);     // s[0 .. w)
    T* hm = sm + w;                             // hh[l0 .. l0 + w + rows + 1)
    T* xm = hm + w + rows + 1;                  // [V][NC w]
    T* sums = xm + V * NC * w;                  // [warp][V][NC]
    for (int i = tid; i < w; i += kThreads) sm[i] = P.s[i];
    for (int i = tid; i < w + rows + 1; i += kThreads) hm[i] = P.hh[l0 + i];
    for (int i = tid; i < NC * w; i += kThreads) {
        const int64_t kp = k0 + (int64_t)NC * a0 + i;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            T x = T(0);
            if (g0 + v < P.batch) x = scaled_input(P, P.in + (g0 + v) * P.n, P.n, kp);
            xm[v * NC * w + i] = x;
        }
    }
    __syncthreads();
    const int r = warp / WR, part = warp % WR;
    T acc[V][NC];
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[v][c] = T(0);
    for (int b = r + lane + 32 * part; b < w; b += 32 * WR) {
        const T s = sm[b - r];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const T e = s * hm[r + b + c];
#pragma unroll
            for (int v = 0; v < V; ++v) acc[v][c] += e * xm[v * NC * w + NC * b + c];
        }
    }
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int k = 16; k > 0; k >>= 1)
                acc[v][c] += __shfl_xor_sync(0xffffffffu, acc[v][c], k);
    T y = T(0);
#pragma unroll
    for (int v = 0; v < V; ++v)
#pragma unroll
        for (int c = 0; c < NC; ++c)
            if (lane == v * NC + c) y = acc[v][c];
    if constexpr (WR > 1) {
        if (lane < NC * V) sums[warp * (NC * V) + lane] = y;
        __syncthreads();
    }
    if (part == 0 && lane < NC * V && a0 + r < m) {
#pragma unroll
        for (int i = 1; i < WR; ++i) y += sums[(warp + i) * (NC * V) + lane];
        const int64_t g = g0 + lane / NC;
        const int64_t kp = k0 + (int64_t)NC * (a0 + r) + lane % NC;
        const int64_t k = P.rev ? P.npk - 1 - kp : kp;
        if (g < P.batch && k < P.n) {
            y *= P.dout[k];
            if (P.sign_out && (k & 1)) y = -y;
            if (k == 0 && P.a00) y += P.a00[0] * P.in[g * P.n];
            P.out[g * P.n + k] = y;
        }
    }
}

// --------------------------------------------------------------------------- ragged lists
//
// Vectors sorted by length, longest first (leaf counts; equal counts in any order: every
// vector's arithmetic is its own), so the vectors a CTA takes together are about as long as
// each other.  Conditions recorded in the status word: the output range overlapping the
// input's (nothing is converted), vectors longer than n_max or with decreasing offsets (left
// unwritten).
constexpr int kSortThreads = 1024;

__device__ __forceinline__ int ragged_bin(const int64_t* offs, int64_t v, int64_t n_max, int unit,
                                          int bins, int* bad) {
    const int64_t n = offs[v + 1] - offs[v];
    if (n < 0 || n > n_max) *bad = 1;
    if (n <= 0 || n > n_max) return -1;
    return bins - (int)((n + unit - 1) / unit);  // 0: the longest
}

__device__ __forceinline__ bool ragged_alias(const int64_t* offs, int64_t batch, const char* in,
                                             const char* out, int esz) {
    const int64_t span = (offs[batch] - offs[0]) * esz;
    const int64_t gap = in > out ? (int64_t)(in - out) : (int64_t)(out - in);
    return span > 0 && gap < span;
}

// hist[bins + 1]: counts per bin (cleared before the launch)
__global__ void k_hier_hist(const int64_t* __restrict__ offs, int64_t batch, int64_t n_max,
                            int unit, int bins, int* __restrict__ hist, const char* in,
                            const char* out, int esz, int* status) {
    if (ragged_alias(offs, batch, in, out, esz)) {
        if (blockIdx.x == 0 && threadIdx.x == 0 && status) atomicOr(status, TDH_STATUS_ALIAS);
        return;
    }
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= batch) return;
    int bad = 0;
    const int b = ragged_bin(offs, v, n_max, unit, bins, &bad);
    if (bad && status) atomicOr(status, TDH_STATUS_LENGTH);
    if (b >= 0) atomicAdd(&hist[b], 1);
}

// exclusive prefix sums in place; hist[bins] = the number of vectors to convert
__global__ void __launch_bounds__(kSortThreads) k_hier_scan(int* __restrict__ hist, int bins) {
    __shared__ int wsum[kSortThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int carry = 0;
    for (int b0 = 0; b0 < bins; b0 += kSortThreads) {
        const int i = b0 + tid;
        const int x = i < bins ? hist[i] : 0;
        int s = x;
        for (int k = 1; k < 32; k <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, s, k);
            if (lane >= k) s += o;
        }
        if (lane == 31) wsum[warp] = s;
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < kSortThreads / 32; ++w) {
            if (w < warp) before += wsum[w];
            total += wsum[w];
        }
        if (i < bins) hist[i] = carry + before + s - x;
        carry += total;
        __syncthreads();
    }
    if (tid == 0) hist[bins] = carry;
}

__global__ void k_hier_scatter(const int64_t* __restrict__ offs, int64_t batch, int64_t n_max,
                               int unit, int bins, int* __restrict__ hist, int* __restrict__ list,
                               const char* in, const char* out, int esz) {
    if (ragged_alias(offs, batch, in, out, esz)) return;
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= batch) return;
    int bad = 0;
    const int b = ragged_bin(offs, v, n_max, unit, bins, &bad);
    if (b >= 0) list[atomicAdd(&hist[b], 1)] = (int)v;
}

// The same in one launch of one CTA (hist[0 .. bins) unused): each launch of the three and the
// clearing of their counts costs 2 to 3 us, more than a few thousand vectors do.  Leg->Cheb float32
// 128 x 512: 24.7 -> 16.9 us, 200 x 512: 31.8 -> 22.1, 512 x 2048: 42.4 -> 33.6 (with one scratch
// block for lists and tree, and the moments' launch overlapping this one); the FFT classes take
// 21.7, 23.5 and 45.2.
constexpr int kSmallSort = 4 * kSortThreads;  // vectors
__global__ void __launch_bounds__(kSortThreads) k_hier_sort(const int64_t* __restrict__ offs,
                                                            int batch, int64_t n_max, int unit,
                                                            int bins, int* __restrict__ hist,
                                                            int* __restrict__ list, const char* in,
                                                            const char* out, int esz, int* status) {
    __shared__ int at[kSortThreads], wsum[kSortThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    pdl_trigger();
    if (ragged_alias(offs, batch, in, out, esz)) {
        if (tid == 0) {
            hist[bins] = 0;
            if (status) atomicOr(status, TDH_STATUS_ALIAS);
        }
        return;
    }
    at[tid] = 0;
    __syncthreads();
    int bin[kSmallSort / kSortThreads], bad = 0;
#pragma unroll
    for (int k = 0; k < kSmallSort / kSortThreads; ++k) {
        const int v = k * kSortThreads + tid;
        bin[k] = v < batch ? ragged_bin(offs, v, n_max, unit, bins, &bad) : -1;
        if (bin[k] >= 0) atomicAdd(&at[bin[k]], 1);
    }
    if (bad && status) atomicOr(status, TDH_STATUS_LENGTH);
    __syncthreads();
    const int x = at[tid];
    int s = x;
    for (int k = 1; k < 32; k <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, s, k);
        if (lane >= k) s += o;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    at[tid] = before + s - x;
    if (tid == kSortThreads - 1) hist[bins] = before + s;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSmallSort / kSortThreads; ++k)
        if (bin[k] >= 0) list[atomicAdd(&at[bin[k]], 1)] = k * kSortThreads + tid;
}

// ------------------------------------------------------------------------------ host side

double lagrange(const int* x, int P, int i, double at) {
    double v = 1.0;
    for (int j = 0; j < P; ++j)
        if (j != i) v *= (at - x[j]) / (double)(x[i] - x[j]);
    return v;
}

// Float32 tables are scaled by constants, so that no rounding is common to all entries, or to the
// leading ones, which dominate decaying inputs: s_0 becomes a power of two (every diagonal entry
// has it) and h takes its mantissa.  Where D1 varies and is inexact anyway, h's first entry on the
// diagonal (index 2 j0) becomes one too and D1, rounded once, takes that; Leg->Cheb's constant D1
// (2/pi) gives its mantissa to h instead; Cheb->Leg's D1 (j + 1/2) is exact and stays.  Float64
// keeps the symbols, which are float64 already.
struct HierScale {
    double s, h, d;  // table = symbol * factor
};
__device__ __forceinline__ double mantissa(double v) {
    if (v == 0.0 || !isfinite(v)) return 1.0;
    int e;
    return fabs(frexp(v, &e)) * 2.0;
}
template <typename T>
__device__ __forceinline__ HierScale hier_scale(const double* t, const double* h, int kind, int j0) {
    if (sizeof(T) == 8) return HierScale{1.0, 1.0, 1.0};
    const double mt = mantissa(t[0]);
    const double md = kind == TDH_LEG2CHEB ? 1.2732395447351628 : 1.0;  // 4/pi
    const double mh =
        kind == TDH_LEG2CHEB || kind == TDH_CHEB2LEG ? 1.0 : mantissa(h[2 * j0] * mt);
    return HierScale{1.0 / mt, mt * md / mh, mh / md};
}

// D1 for the tables below
template <typename T>
__global__ void k_hier_diagonal(const double* __restrict__ t, const double* __restrict__ h,
                                const double* __restrict__ d1, int kind, int j0, int64_t n,
                                T* __restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < n) out[i] = (T)(d1[i] * hier_scale<T>(t, h, kind, j0).d);
}

// table copies in execute precision: s_m = t[stride m] (32 zeros before, zero past mpad),
// hf_l = h[stride l], hr_i = hf[2 mrev - 1 - i] (zero past 2 mrev); entry 0 of h dropped where
// (0, 0) is direct
template <typename T>
__global__ void k_hier_tables(const double* __restrict__ t, const double* __restrict__ h,
                              int kind, int64_t mpad, int64_t mrev, int stride, int j0,
                              T* __restrict__ s, T* __restrict__ hf, T* __restrict__ hr) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    const HierScale c = hier_scale<T>(t, h, kind, j0);
    if (i < kHierSZero) s[i - kHierSZero] = T(0);
    if (i < mpad) s[i] = (T)(t[stride * i] * c.s);
    if (i < 2 * mpad + kHierHPad) {
        const T v = (i >= 2 * mpad || (j0 == 1 && i == 0)) ? T(0) : (T)(h[stride * i] * c.h);
        hf[i] = v;
        if (i < 2 * mrev)
            hr[2 * mrev - 1 - i] = v;
        else
            hr[i] = T(0);
    }
}

// s at the points of the 2048-boxes, [distance][P][P], then h forward and reversed,
// [sum of indices][NC][P][P].
template <typename T>
__global__ void k_hier_points(const T* __restrict__ s, const T* __restrict__ hf,
                              const T* __restrict__ hr, int nc, int64_t ns, int64_t nh,
                              T* __restrict__ out) {
    constexpr int P = HierP<T>::P, TOP = kHierLevels - 1;
    __shared__ int x[P];
    if (threadIdx.x == 0)
#pragma unroll
        for (int i = 0; i < P; ++i) x[i] = hier_point<P>(TOP, i);
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= ns + 2 * nh) return;
    const int xq = x[i % P], xp = x[i / P % P];  // every table is whole [P][P] blocks
    if (i < ns) {
        const int64_t at = i / (P * P) * kHierTop + xq - xp;
        out[i] = at >= 0 ? s[at] : T(0);
    } else {
        const bool rev = i >= ns + nh;
        const int64_t b = (i - ns - (rev ? nh : 0)) / (P * P);
        out[i] = (rev ? hr : hf)[b / nc * kHierTop + xp + xq + b % nc];
    }
}

// Packed length of a reversed vector of m indices: whole boxes of the largest size that exchanges
// anything (three boxes or more), so that its last one ends at index 0, beyond which h is not
// smooth, and the padding lies before its first leaf.  (Whole 2048-boxes for every length made
// transposes of short vectors form moments and launch warps for up to 63 empty leaves: Leg->Cheb
// 200 x 1024 float32 41 us, now 18; the FFTs take 29.)
int64_t reversed_length(int64_t m) {
    int l = kHierLevels - 1;
    while (l > 0 && m <= 2 * hier_size(l)) --l;
    return (m + hier_size(l) - 1) / hier_size(l) * hier_size(l);
}

template <typename T>
int prepare_typed(Step& st, cudaStream_t s) {
    constexpr int P = HierP<T>::P;
    HierData& H = st.hier;
    const int NC = st.full ? 1 : 2;
    H.mpad = (hier_length(st) - 2) / NC;
    H.mrev = reversed_length((st.n + NC - 1) / NC);
    const size_t ns = (size_t)(H.mpad + kHierSZero), nh = (size_t)(2 * H.mpad + kHierHPad);
    const size_t nw = (size_t)P * kHierLeaf + 12 * P * P;
    // long vectors: the 2048-boxes' point tables (k_hier_top)
    const int64_t ntop = H.mpad / kHierTop;
    const bool top = ntop >= kTopKernel;
    const int64_t nps = top ? ntop * P * P : 0, nph = top ? (2 * ntop - 1) * NC * P * P : 0;
    const size_t at = (ns + 2 * nh + nw + 3) / 4 * 4;  // 16-byte aligned
    int rc = dev_alloc(&H.tab, sizeof(T) * (at + (size_t)(nps + 2 * nph)));
    std::vector<T> w(nw);
    if (rc == TDH_OK) {
        T* tab = static_cast<T*>(H.tab);
        H.s = tab + kHierSZero;
        H.hf = tab + ns;
        H.hr = tab + ns + nh;
        H.w = tab + ns + 2 * nh;
        cudaError_t e = cudaSuccess;
        H.d1 = st.d1x;
        if (sizeof(T) == 4) {
            // formed where the Hankel table will be, then kept in place of the float64 D1, which
            // nothing reads any more (an allocation of its own: 50 us more per one-off conversion)
            k_hier_diagonal<T><<<(unsigned)((st.n + kThreads - 1) / kThreads), kThreads, 0, s>>>(
                st.t, st.h, st.d1, st.kind, (int)st.j0, st.n, static_cast<T*>(H.hf));
            e = cudaMemcpyAsync(st.d1, H.hf, sizeof(T) * (size_t)st.n, cudaMemcpyDeviceToDevice, s);
            H.d1 = st.d1;
        }
        const int64_t cnt = 2 * H.mpad + kHierHPad;
        k_hier_tables<T><<<(unsigned)((cnt + kThreads - 1) / kThreads), kThreads, 0, s>>>(
            st.t, st.h, st.kind, H.mpad, H.mrev, NC, (int)st.j0, static_cast<T*>(H.s),
            static_cast<T*>(H.hf), static_cast<T*>(H.hr));
        if (top) {
            H.st = tab + at;
            H.ht[0] = tab + at + nps;
            H.ht[1] = tab + at + nps + nph;
            // (reversed full kinds start one entry on, as in run_typed)
            k_hier_points<T><<<(unsigned)((nps + 2 * nph + kThreads - 1) / kThreads), kThreads, 0, s>>>(
                static_cast<const T*>(H.s), static_cast<const T*>(H.hf),
                static_cast<const T*>(H.hr) + (NC == 1 ? 1 : 0), NC, nps, nph, tab + at);
        }
        int x[kHierLevels][P];
        for (int l = 0; l < kHierLevels; ++l)
            for (int p = 0; p < P; ++p) x[l][p] = hier_point<P>(l, p);
        for (int p = 0; p < P; ++p)
            for (int a = 0; a < kHierLeaf; ++a)
                w[(size_t)p * kHierLeaf + a] = (T)lagrange(x[0], P, p, a);
        for (int l = 1; l < kHierLevels; ++l)
            for (int c = 0; c < 4; ++c)
                for (int p = 0; p < P; ++p)
                    for (int q = 0; q < P; ++q)
                        w[(size_t)P * kHierLeaf + (((l - 1) * 4 + c) * P + p) * P + q] =
                            (T)lagrange(x[l], P, p, c * hier_size(l - 1) + x[l - 1][q]);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(H.w, w.data(), sizeof(T) * nw, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            set_error("hierarchical tables: %s", cudaGetErrorString(e));
            rc = TDH_ERR_CUDA;
        }
    }
    if (rc == TDH_OK) H.on = H.use = 1;
    H.use_ragged = H.use && NC == 2;
    return rc;
}

template <typename T, int NC, int NVT>
size_t far_smem(int SL) {
    using F = FarShape<T, NC, NVT>;
    size_t boxes = kTopSplit;
    for (int l = 0; l < kHierLevels - 1; ++l) boxes += std::max(1, SL >> (2 * l));
    return sizeof(T) * (kHierSZero + 8 * kHierLeaf + 2 * SL * kHierLeaf + 10 * kHierLeaf + F::trw +
                        (SL + 7) * NC * F::VTL * F::MG + boxes * F::erow);
}

template <typename T, int NC, int NV, bool RAGGED>
constexpr size_t near_smem() {
    using S = NearShape<T, NC, NV>;
    return 2 * sizeof(T) * (size_t)(S::table_pairs + S::warps * S::warp_pairs(RAGGED));
}

template <typename T>
size_t up_smem(int NC, int NVT) {
    constexpr int P = HierP<T>::P;
    constexpr int VW = 32 / P;
    return sizeof(T) * ((size_t)kWarps * VW * (NC * kHierLeaf + 16 / sizeof(T)) +
                        (size_t)(kHierTopLeaves + kHierTopLeaves / 4 + kHierTopLeaves / 16) * NC *
                            NVT * P +
                        (size_t)12 * P * P);
}

constexpr size_t kMaxSmem = 227 * 1024;

template <typename T>
cudaError_t launch_cfg(void (*kern)(const HierParams<T>), unsigned grid, size_t smem,
                       cudaStream_t s, bool pdl, const HierParams<T>& P,
                       int threads = kThreads) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute a[1];
    a[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, P);
}

template <typename T, int NC, bool RAGGED>
int launch_up(const HierParams<T>& P, unsigned grid, cudaStream_t s) {
    // dense: launched without overlap, as its input may be the previous step's output (ragged: it
    // waits for the lists, whose kernels are launched without)
    auto kern = k_hier_up<T, NC, RAGGED>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem);
    });
    if (e == cudaSuccess) e = launch_cfg<T>(kern, grid, up_smem<T>(NC, P.unvt), s, RAGGED && P.first == 0, P);
    if (e != cudaSuccess) {
        set_error("hierarchical moments: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, int NVT, bool RAGGED>
int launch_far(const HierParams<T>& P, unsigned grid, cudaStream_t s) {
    auto kern = k_hier_far<T, NC, NVT, RAGGED>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem - 1024);
    });
    if (e == cudaSuccess)
        e = launch_cfg<T>(kern, grid, far_smem<T, NC, NVT>(P.seg_leaves), s, true, P);
    if (e != cudaSuccess) {
        set_error("hierarchical far field: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, int NVT, bool RAGGED>
int launch_top(const HierParams<T>& P, unsigned grid, cudaStream_t s) {
    const cudaError_t e = launch_cfg<T>(k_hier_top<T, NC, NVT, RAGGED>, grid, 0, s, true, P);
    if (e != cudaSuccess) {
        set_error("hierarchical far field: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, int NV, bool REV, bool RAGGED>
int launch_near_rev(const HierParams<T>& P, unsigned grid, bool pdl, cudaStream_t s) {
    constexpr size_t smem = near_smem<T, NC, NV, RAGGED>();
    static_assert(smem <= kMaxSmem, "shared memory budget");
    auto kern = k_hier_near<T, NC, NV, REV, RAGGED>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    if (e == cudaSuccess)
        e = launch_cfg<T>(kern, grid, smem, s, pdl, P, 32 * NearShape<T, NC, NV>::warps);
    if (e != cudaSuccess) {
        set_error("hierarchical near field: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, int NV, bool RAGGED>
int launch_near_nv(const HierParams<T>& P, int64_t nb, bool pdl, cudaStream_t s) {
    const int64_t tasks = (nb + NV - 1) / NV * P.runs;
    constexpr int W = NearShape<T, NC, NV>::warps;
    const unsigned grid = (unsigned)((tasks + W - 1) / W);
    if constexpr (!RAGGED)
        if (P.rev) return launch_near_rev<T, NC, NV, true, false>(P, grid, pdl, s);
    return launch_near_rev<T, NC, NV, false, RAGGED>(P, grid, pdl, s);
}

template <typename T, int NC, bool RAGGED>
int launch_near(const HierParams<T>& P, int NV, int64_t nb, bool pdl, cudaStream_t s) {
    constexpr int VMAX = sizeof(T) == 4 ? 32 : 16;
    if (NV == VMAX) return launch_near_nv<T, NC, VMAX, RAGGED>(P, nb, pdl, s);
    if (NV == 16) return launch_near_nv<T, NC, 16, RAGGED>(P, nb, pdl, s);
    if (NV == 8) return launch_near_nv<T, NC, 8, RAGGED>(P, nb, pdl, s);
    return launch_near_nv<T, NC, 2, RAGGED>(P, nb, pdl, s);
}

// The direct product's shared memory, the vectors a CTA takes (0: too long for it), and whether it
// is the faster way.
template <typename T>
size_t direct_smem(int NC, int64_t m, int V) {
    return sizeof(T) * (size_t)(2 * m + kWarps + 1 + V * NC * (m + kWarps));
}
template <typename T>
int direct_vectors(int NC, int64_t m, int64_t batch) {
    int V = batch == 1 ? 1 : batch == 2 ? 2 : 4;
    while (V > 0 && direct_smem<T>(NC, m, V) > kMaxSmem) V = V == 4 ? 2 : 0;
    return V;
}
template <typename T>
bool direct_serves(int NC, int64_t m, int64_t batch) {
    const int V = direct_vectors<T>(NC, m, batch);
    if (V == 0) return false;
    // Lane operations: multiply-adds, the entries' products among them, half a warp of each row
    // idle on average, and a row's reductions (five adds a lane and sum); against the tree, whose
    // few launches take about the same time for any short vectors (float32 21 us, Jacobi 16;
    // float64 185 and 125 us), or its one launch where there is no far field (two leaves: float32
    // 6 to 9 us, float64 60 to 100).  Measured, direct: float64 113 us at 45e6 (Leg->Cheb 5700 x 4),
    // 60 us at 21e6 (100 x 1000), 114 us at 52e6 (64 x 4096, the tree 63); float32 Leg->Cheb
    // 15.4 us at 31e6 (1000 x 64, the tree 19.4), 19.3 us at 48e6 (4096 x 8, the tree 25.2 and the
    // FFTs 23.9), 25.6 us at 49e6 (6000 x 4, 24.3), 23.6 us at 63e6 (1000 x 128, 19.9); Jacobi
    // 17.4 us at 39e6 (1000 x 48, 18.9), 19.4 us at 49e6 (200 x 800, 18.2).
    const double cost = NC * (double)m * (double)((batch + V - 1) / V) *
                        ((V + 1) * (0.5 * (double)m + 16) + 160 * V);
    if (m <= 2 * kHierLeaf) return cost <= (sizeof(T) == 4 ? 14.5e6 : 22e6);
    return cost <= (sizeof(T) == 4 ? (NC == 2 ? 48e6 : 40e6) : NC == 2 ? 70e6 : 44e6);
}

template <typename T, int NC, int V, int WR>
int launch_direct_wr(const HierParams<T>& P, int64_t m, unsigned grid, cudaStream_t s) {
    auto kern = k_hier_direct<T, NC, V, WR>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem);
    });
    if (e == cudaSuccess) {
        kern<<<(unsigned)grid, kThreads, direct_smem<T>(NC, m, V), s>>>(P, (int)m);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("direct product: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

// Rows per CTA (8 / WR) halved until every SM has a CTA: the SM that holds the longest rows sets
// the time, in float64 by its 2 multiply-adds per clock (Leg->Cheb n = 1024 float64: 10.4 us with
// 64 CTAs of 8 rows, 7.5 us with 256 of 2).
template <typename T, int NC, int V>
int launch_direct(const HierParams<T>& P, int64_t m, cudaStream_t s) {
    const int64_t groups = (P.batch + V - 1) / V;
    auto grid = [&](int rows) { return (m + rows - 1) / rows * groups; };
    if (grid(8) >= sm_count()) return launch_direct_wr<T, NC, V, 1>(P, m, (unsigned)grid(8), s);
    if (grid(4) >= sm_count()) return launch_direct_wr<T, NC, V, 2>(P, m, (unsigned)grid(4), s);
    return launch_direct_wr<T, NC, V, 4>(P, m, (unsigned)grid(2), s);
}

// Lists of a ragged batch, into scr: hist[bins + 1], then list[batch].
constexpr int kRaggedUnit = 2 * kHierLeaf;  // coefficients of a leaf (two channels)

template <typename T>
int ragged_lists(const Step& st, const void* in, void* out, const int64_t* offs, int64_t batch,
                 int bins, int* scr, cudaStream_t s) {
    int* list = scr + bins + 1;
    cudaError_t e = cudaSuccess;
    const unsigned grid = (unsigned)((batch + kThreads - 1) / kThreads);
    const char* ci = static_cast<const char*>(in);
    const char* co = static_cast<const char*>(out);
    if (batch <= kSmallSort && bins <= kSortThreads) {
        k_hier_sort<<<1, kSortThreads, 0, s>>>(offs, (int)batch, st.n, kRaggedUnit, bins, scr, list,
                                               ci, co, (int)sizeof(T), st.status);
        note_launches(1);
        e = cudaGetLastError();
    } else {
        e = cudaMemsetAsync(scr, 0, sizeof(int) * (size_t)(bins + 1), s);
        if (e == cudaSuccess) {
            k_hier_hist<<<grid, kThreads, 0, s>>>(offs, batch, st.n, kRaggedUnit, bins, scr, ci, co,
                                                  (int)sizeof(T), st.status);
            k_hier_scan<<<1, kSortThreads, 0, s>>>(scr, bins);
            k_hier_scatter<<<grid, kThreads, 0, s>>>(offs, batch, st.n, kRaggedUnit, bins, scr, list,
                                                     ci, co, (int)sizeof(T));
            note_launches(3);
            e = cudaGetLastError();
        }
    }
    if (e != cudaSuccess) {
        set_error("ragged lists: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    return TDH_OK;
}

template <typename T, int NC, bool RAGGED>
int run_typed(const Step& st, const void* in, void* out, const int64_t* offs, int64_t batch,
              int adjoint, cudaStream_t s) {
    constexpr int NP = HierP<T>::P;
    const HierData& H = st.hier;
    const int64_t m = (st.n + NC - 1) / NC;
    HierParams<T> P{};
    P.n = st.n;
    P.npk = NC * (adjoint ? H.mrev : H.mpad);
    P.s = static_cast<const T*>(H.s);
    // reversed: packed index a' + b' meets hf[2 (mrev - 1) - a' - b' (+ 1 in channel 0)]
    P.hh = static_cast<const T*>(adjoint ? H.hr : H.hf) + (adjoint && NC == 1 ? 1 : 0);
    P.st = static_cast<const T*>(H.st);
    P.ht = static_cast<const T*>(H.ht[adjoint ? 1 : 0]);
    P.lw = static_cast<const T*>(H.w);
    P.tr = P.lw + NP * kHierLeaf;
    P.din = static_cast<const T*>(adjoint ? H.d1 : st.d2x);
    P.dout = static_cast<const T*>(adjoint ? st.d2x : H.d1);
    P.a00 = st.j0 == 1 ? static_cast<const T*>(st.row0) : nullptr;
    P.rev = adjoint;
    P.aligned = st.n * (int64_t)sizeof(T) % 16 == 0;
    P.sign_in = st.sign_in;
    P.sign_out = st.sign_out;
    if (adjoint) {
        P.leaf0 = (int)((H.mrev - m) / kHierLeaf);
        P.leaves = (int)(H.mrev / kHierLeaf);
    } else {
        P.leaf0 = 0;
        P.leaves = (int)((m + kHierLeaf - 1) / kHierLeaf);
    }
    const int64_t real_leaves = (m + kHierLeaf - 1) / kHierLeaf;
    if (!RAGGED && direct_serves<T>(NC, m, batch)) {
        P.batch = batch;
        P.in = static_cast<const T*>(in);
        P.out = static_cast<T*>(out);
        const int V = direct_vectors<T>(NC, m, batch);
        return V == 1   ? launch_direct<T, NC, 1>(P, m, s)
               : V == 2 ? launch_direct<T, NC, 2>(P, m, s)
                        : launch_direct<T, NC, 4>(P, m, s);
    }
    // vectors of a near-field warp, and of a far-field CTA
    constexpr int VMAX = sizeof(T) == 4 ? 32 : 16;
    constexpr int FMAX = sizeof(T) == 4 ? 16 : 8;
    P.seg_leaves = real_leaves > 4 ? 16 : 4;
    P.nseg = (P.leaves + P.seg_leaves - 1) / P.seg_leaves;
    // Two vectors per far CTA while such CTAs do not fill the chip, as a CTA's time grows with its
    // vectors (Leg->Cheb 16000 x 8 float64: 343 us with 8, 188 us with 2, the near field's vectors
    // chosen alike), else FMAX: nothing between, so just past the switch grids are small (65536 x 5
    // float32: 64 CTAs) and slots empty.
    P.nvt = batch > 2 && (batch + 1) / 2 * P.nseg > sm_count() ? FMAX : 2;
    P.unvt = 32 / NP;
    // Near field: vectors of a warp (twice as many on half as many warps do the same work per SM
    // and step with fewer loads, about 15 % less time) and leaves it walks (a walk loads one leaf
    // more than it completes).  One CTA per SM is resident: the waves should be full.
    int NV = 2;
    double best = 0;
    for (int nv = 2; nv <= VMAX; nv *= nv == 2 ? 4 : 2) {
        const int64_t slots = (nv == VMAX ? 8 : 16) * (int64_t)sm_count();
        const int64_t vgroups = (batch + nv - 1) / nv;
        const double step = nv == VMAX ? 1.0
                            : nv == 2  ? 0.65
                            : nv == 16 || sizeof(T) == 8 ? 1.15 * nv / (VMAX / 2) : 0.8;
        for (int run = 16; run >= 1; --run) {
            const int64_t tasks = (real_leaves + run - 1) / run * vgroups;
            const double cost = (double)((tasks + slots - 1) / slots) * (run + 0.4) * step;
            if (best == 0 || cost < best) {
                best = cost;
                P.run = run;
                NV = nv;
            }
        }
        if (batch <= 2) break;
    }
    P.runs = (real_leaves + P.run - 1) / P.run;
    const int64_t ntop = (P.leaves + kHierTopLeaves - 1) / kHierTopLeaves;
    // moments of every box and expansions of every leaf of a vector; about 1 GB at a time
    int64_t boxes[kHierLevels], total = 0;
    for (int l = 0; l < kHierLevels; ++l)
        total += boxes[l] = (P.leaves + (1 << (2 * l)) - 1) >> (2 * l);
    const bool far = real_leaves > 2;
    P.ntop = (int)ntop;
    const bool top = ntop >= kTopKernel;
    const int64_t per_vec =
        (total + boxes[0] + (top ? ntop : 0)) * NC * NP * (int64_t)sizeof(T);
    const int unit = std::max(std::max(P.nvt, P.unvt), NV);  // powers of two
    int64_t chunk = std::max<int64_t>(1, ((int64_t)1 << 30) / per_vec);
    chunk = std::min(chunk, (int64_t)INT32_MAX / 4 / std::max<int64_t>(P.runs, ntop));
    chunk = std::max<int64_t>(unit, chunk / unit * unit);
    chunk = std::min<int64_t>(chunk, (batch + unit - 1) / unit * unit);
    // one block: the lists of a ragged batch, then the moments and expansions
    const int bins = RAGGED ? (int)((st.n + kRaggedUnit - 1) / kRaggedUnit) : 0;
    const size_t head =
        RAGGED ? (sizeof(int) * (size_t)(bins + 1 + batch) + 255) / 256 * 256 : 0;
    char* scr = nullptr;
    if (RAGGED || far)
        for (;;) {  // (fewer vectors at a time where memory is short)
            const int rc = scratch_alloc(reinterpret_cast<void**>(&scr),
                                         head + (far ? (size_t)(per_vec * chunk) : 0), s);
            if (rc == TDH_OK) break;
            if (rc != TDH_ERR_NOMEM || !far || chunk <= unit ||
                (size_t)(per_vec * chunk) <= kLeastScratch)
                return rc;
            chunk = std::max<int64_t>(unit, chunk / 2 / unit * unit);
        }
    const int* list = reinterpret_cast<const int*>(scr) + bins + 1;
    T* mom = far ? reinterpret_cast<T*>(scr + head) : nullptr;
    P.bpad = chunk;
    for (int l = 0; l < kHierLevels; ++l) {
        P.mom[l] = mom;
        if (mom) mom += boxes[l] * NC * NP * chunk;
    }
    P.loc = mom;
    P.top = top ? mom + boxes[0] * NC * NP * chunk : nullptr;
    int rc = TDH_OK;
    if constexpr (RAGGED)
        rc = ragged_lists<T>(st, in, out, offs, batch, bins, reinterpret_cast<int*>(scr), s);
    for (int64_t b0 = 0; rc == TDH_OK && b0 < batch; b0 += chunk) {
        const int64_t nb = std::min(chunk, batch - b0);
        P.batch = nb;
        P.in = static_cast<const T*>(in);
        P.out = static_cast<T*>(out);
        if constexpr (RAGGED) {
            P.offs = offs;
            P.list = list + b0;
            P.first = b0;
            P.count = list - 1;
        } else {
            P.in += b0 * st.n;
            P.out += b0 * st.n;
        }
        if (far) {
            const int64_t groups = (nb + P.nvt - 1) / P.nvt;
            rc = launch_up<T, NC, RAGGED>(
                P, (unsigned)((groups * P.nvt + P.unvt - 1) / P.unvt * ntop), s);
            const unsigned grid = (unsigned)(groups * P.nseg);
            if (rc == TDH_OK && top)
                rc = P.nvt == FMAX
                         ? launch_top<T, NC, FMAX, RAGGED>(P, (unsigned)(groups * ntop), s)
                         : launch_top<T, NC, 2, RAGGED>(P, (unsigned)(groups * ntop), s);
            if (rc == TDH_OK)
                rc = P.nvt == FMAX ? launch_far<T, NC, FMAX, RAGGED>(P, grid, s)
                                   : launch_far<T, NC, 2, RAGGED>(P, grid, s);
        }
        if (rc == TDH_OK) rc = launch_near<T, NC, RAGGED>(P, NV, nb, far, s);
    }
    scratch_free(scr, s);
    return rc;
}

}  // namespace

// The boxes at the end reach past n: whole 2048-boxes per channel.
int64_t hier_length(const Step& st) {
    const int NC = st.full ? 1 : 2;
    const int64_t m = (st.n + NC - 1) / NC;
    return NC * ((m + kHierTop - 1) / kHierTop * kHierTop) + 2;
}

int hier_prepare(Step& st, int prec, cudaStream_t s) {
    return prec != TDH_FP64 ? prepare_typed<float>(st, s) : prepare_typed<double>(st, s);
}

void hier_release(HierData& h) {
    dev_free(h.tab);
    h = HierData{};
}

int hier_launch(const Step& st, int prec, const void* in, void* out, int64_t batch, int adjoint,
                cudaStream_t s) {
    if (prec != TDH_FP64)
        return st.full ? run_typed<float, 1, false>(st, in, out, nullptr, batch, adjoint, s)
                       : run_typed<float, 2, false>(st, in, out, nullptr, batch, adjoint, s);
    return st.full ? run_typed<double, 1, false>(st, in, out, nullptr, batch, adjoint, s)
                   : run_typed<double, 2, false>(st, in, out, nullptr, batch, adjoint, s);
}

int hier_launch_ragged(const Step& st, int prec, const void* in, void* out, const int64_t* offs,
                       int64_t batch, cudaStream_t s) {
    return prec != TDH_FP64 ? run_typed<float, 2, true>(st, in, out, offs, batch, 0, s)
                            : run_typed<double, 2, true>(st, in, out, offs, batch, 0, s);
}

}  // namespace tdh
