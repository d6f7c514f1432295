// Kernels and host side of the hierarchical T o H product (tdh_hier.cuh).
//
// Two launches per step: k_hier_up forms the moments of every box, k_hier_down exchanges them,
// passes the local expansions down and adds the near field.  Vectors are independent; a CTA
// takes a segment of rows of a few vectors, so every table entry it forms serves all of them.
#include <algorithm>
#include <cmath>
#include <vector>

#include "tdh_hier.cuh"

namespace tdh {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kTopSplit = 8;  // ways the 2048-boxes' exchange is split over a CTA's threads

template <typename T>
struct HierParams {
    static constexpr int P = HierP<T>::P;
    const T* in;
    T* out;
    int64_t n;       // coefficients per vector (dense)
    int64_t npk;     // NC * mpad: padded length (index reversal)
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
    int nseg, seg_leaves, nvt, unvt;  // down-kernel segments; vectors per CTA (down, up)
    short x[kHierLevels][P];
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
};
template <>
struct Vec16<double> {
    static constexpr int N = 2;
    double v[2];
    __device__ __forceinline__ void load(const double* p) {
        const double2 q = *reinterpret_cast<const double2*>(p);
        v[0] = q.x, v[1] = q.y;
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

// ------------------------------------------------------------------------------- moments
//
// A CTA forms the moments of one 2048-box (64 leaves, their parents, ...) for unvt vectors.  A
// warp takes one leaf of VW vectors at a time: lane (p, v) holds the 32 weights L_p in
// registers, so each 16-byte shared load of inputs feeds 16 bytes' worth of multiply-adds.
template <typename T, int NC, bool RAGGED>
__global__ void __launch_bounds__(kThreads) k_hier_up(const __grid_constant__ HierParams<T> P) {
    constexpr int NP = HierP<T>::P;
    constexpr int VW = 32 / NP;
    constexpr int XW = NC * kHierLeaf;                 // inputs of a leaf
    constexpr int XS = XW + 16 / (int)sizeof(T);       // padded row
    constexpr int QV = Vec16<T>::N;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
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
    const int p = lane % NP, vq = lane / NP;
    T lw[kHierLeaf];
#pragma unroll
    for (int a = 0; a < kHierLeaf; ++a) lw[a] = P.lw[p * kHierLeaf + a];
    const int gu = P.unvt / VW;  // vector groups per leaf
    const int64_t boxrow = (int64_t)NC * P.bpad * NP;
    for (int item = warp; item < nl4 * gu; item += kWarps) {
        const int li = item / gu, gv = item % gu;
        const int leaf = l0 + li;
        T acc[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[c] = T(0);
        if (leaf >= P.leaf0 && li < nl) {
            __syncwarp();
#pragma unroll
            for (int v = 0; v < VW; ++v) {
                int64_t base, len;
                vector_at<T, RAGGED>(P, g0 + gv * VW + v, &base, &len);
                const T* x = P.in + base;
#pragma unroll
                for (int i = 0; i < NC; ++i)
                    xw[v * XS + lane + 32 * i] =
                        scaled_input(P, x, len, (int64_t)leaf * XW + lane + 32 * i);
            }
            __syncwarp();
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
            ms0[(size_t)li * row + (c * P.unvt + gv * VW + vq) * NP + p] = acc[c];
            if (li < nl)
                P.mom[0][leaf * boxrow + ((int64_t)c * P.bpad + g0 + gv * VW + vq) * NP + p] =
                    acc[c];
        }
    }
    // parents from children, level by level
    int nb = nl4 / 4;
    const T* src = ms0;
    T* dst = ms1;
    for (int l = 1; l < kHierLevels; ++l) {
        __syncthreads();
        const int nbp = l < kHierLevels - 1 ? (nb + 3) & ~3 : nb;
        for (int i = tid; i < nbp * row; i += kThreads) {
            const int box = i / row, e = i % row;
            const int pp = e % NP, cv = e / NP;
            T acc = T(0);
            if (box < nb) {
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    const T* m = src + (size_t)(4 * box + c) * row + cv * NP;
                    const T* w = P.tr + (((l - 1) * 4 + c) * NP + pp) * NP;
#pragma unroll
                    for (int q = 0; q < NP; q += QV) {
                        Vec16<T> mv, wv;
                        mv.load(m + q);
                        wv.load(w + q);
#pragma unroll
                        for (int j = 0; j < QV; ++j) acc += wv.v[j] * mv.v[j];
                    }
                }
                const int64_t gb = (l0 >> (2 * l)) + box;
                const int c = cv / P.unvt, v = cv % P.unvt;
                P.mom[l][gb * boxrow + ((int64_t)c * P.bpad + g0 + v) * NP + pp] = acc;
            }
            if (l < kHierLevels - 1) dst[(size_t)box * row + e] = acc;
        }
        src = dst;
        dst = ms2;
        nb = nbp / 4;
    }
}

// ------------------------------------------------------------------- exchange, near field
//
// A CTA computes the rows of one segment (seg_leaves leaves: 64, 16, 4 or 1) of nvt vectors:
// the exchange of the segment's boxes (and of the boxes above it, on its path), the local
// expansions down to its leaves, the near field, and the scaled output.
//
// Near field: a warp takes one leaf of NV vectors; the two half-warps take half of the
// vectors each, a lane rows r and r + 16, so each 16-byte broadcast of inputs feeds eight
// multiply-adds, and the entries s h (formed per lane) serve all of the half-warp's vectors.
template <typename T, int NC, int NV, bool RAGGED>
__global__ void __launch_bounds__(kThreads, 2) k_hier_down(const __grid_constant__ HierParams<T> P) {
    constexpr int NP = HierP<T>::P;
    constexpr int QV = Vec16<T>::N;
    constexpr int KV = NV / 2;                 // vectors per half-warp
    constexpr int VPT = NV < 4 ? NV : 4;       // vectors per thread of the exchange
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int xn[kHierLevels][NP];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nseg = P.nseg, SL = P.seg_leaves, NVT = P.nvt;
    const int seg = blockIdx.x % nseg;
    const int64_t g0 = (int64_t)(blockIdx.x / nseg) * NVT;
    const int leaves = group_leaves<T, NC, RAGGED>(P, g0);
    const int l0 = seg * SL;
    if (l0 >= leaves || l0 + SL <= P.leaf0) {
        pdl_wait();  // the launch must not complete before the moments' does
        return;
    }
    const int a0 = l0 * kHierLeaf;
    const int XW = NC * (SL + 1) * kHierLeaf;  // inputs staged: the segment and one leaf more
    const int XS = XW + 16 / (int)sizeof(T);
    // shared memory: inputs, s window [-32, 256), h window, leaf weights, expansions
    T* xs = reinterpret_cast<T*>(smem_raw);
    T* sw = xs + (size_t)NVT * XS + kHierSZero;
    constexpr int SW = 8 * kHierLeaf;
    T* hw = sw + SW;
    const int HW = 2 * SL * kHierLeaf + 10 * kHierLeaf;
    T* lw = hw + HW;                           // [P][32]
    const int erow = NC * NVT * NP;
    int nloc[kHierLevels];                     // boxes of the segment (or its path) per level
    T* ex[kHierLevels];
    {
        T* e = lw + NP * kHierLeaf;
        for (int l = kHierLevels - 1; l >= 0; --l) {
            nloc[l] = max(1, SL >> (2 * l));
            ex[l] = e;
            e += (size_t)(l == kHierLevels - 1 ? kTopSplit : nloc[l]) * erow;
        }
    }
    // the launch's first vector group decides the boxes in play
    if (tid < kHierLevels * NP) xn[tid / NP][tid % NP] = P.x[tid / NP][tid % NP];
    for (int i = tid; i < SW + kHierSZero; i += kThreads) sw[i - kHierSZero] = P.s[i - kHierSZero];
    for (int i = tid; i < HW; i += kThreads) {
        const int64_t g = 2 * (int64_t)a0 + i;
        hw[i] = g < 2 * (P.npk / NC) + kHierHPad - 1 ? P.hh[g] : T(0);
    }
    for (int i = tid; i < NP * kHierLeaf; i += kThreads) lw[i] = P.lw[i];
    for (int i = tid; i < XW; i += kThreads) {
        const int64_t kp = (int64_t)NC * a0 + i;
        const int64_t k = P.rev ? P.npk - 1 - kp : kp;
        T d = T(0);
        if (k >= 0 && (RAGGED || k < P.n)) {
            // ragged: k may pass the tables' end in the last leaf; no vector reaches it
            d = k < P.n ? P.din[k] : T(0);
            if (P.sign_in && (k & 1)) d = -d;
        }
#pragma unroll 4
        for (int v = 0; v < NVT; ++v) {
            int64_t base, len;
            vector_at<T, RAGGED>(P, g0 + v, &base, &len);
            xs[(size_t)v * XS + i] = (k >= 0 && k < len) ? P.in[base + k] * d : T(0);
        }
    }
    __syncthreads();
    // ---- exchange: every level's boxes at once
    const int64_t boxrow = (int64_t)NC * P.bpad * NP;
    const int vts = NVT / VPT;
    pdl_wait();  // the moments were written by the previous kernel
    if (leaves > 2) {
        for (int l = kHierLevels - 1; l >= 0; --l) {
            const bool topl = l == kHierLevels - 1;
            const int size = hier_size(l);
            const int nb = (leaves + (1 << (2 * l)) - 1) >> (2 * l);
            const int split = topl ? kTopSplit : 1;
            const int per = vts * NC * NP;
            const int items = nloc[l] * split * per;
            for (int it = tid; it < items; it += kThreads) {
                const int p = it % NP;
                const int vt = (it / NP) % vts;
                const int c = (it / (NP * vts)) % NC;
                const int bs = it / per;
                const int bl = topl ? 0 : bs;
                const int sp = topl ? bs : 0;
                const int i = (l0 >> (2 * l)) + bl;
                const int xp = xn[l][p];
                T acc[VPT];
#pragma unroll
                for (int u = 0; u < VPT; ++u) acc[u] = T(0);
                const int d1 = topl ? nb - i : min(8 - (i & 3), nb - i);
                const T* mrow = P.mom[l] + ((int64_t)c * P.bpad + g0 + vt * VPT) * NP;
                for (int d = 2 + sp; d < d1; d += split) {
                    const T* m = mrow + (int64_t)(i + d) * boxrow;
                    const T* sp0 = (l == 0 ? sw : P.s) + d * size - xp;
                    const T* hp0 = (l == 0 ? hw + (2 * bl + d) * size
                                           : P.hh + (int64_t)(2 * i + d) * size) + xp + c;
#pragma unroll
                    for (int q0 = 0; q0 < NP; q0 += QV) {
                        T cf[QV];
#pragma unroll
                        for (int j = 0; j < QV; ++j) {
                            const int x = xn[l][q0 + j];
                            cf[j] = sp0[x] * hp0[x];
                        }
#pragma unroll
                        for (int u = 0; u < VPT; ++u) {
                            Vec16<T> mv;
                            mv.load(m + u * NP + q0);
#pragma unroll
                            for (int j = 0; j < QV; ++j) acc[u] += cf[j] * mv.v[j];
                        }
                    }
                }
                T* e = ex[l] + (size_t)bs * erow + (c * NVT + vt * VPT) * NP + p;
#pragma unroll
                for (int u = 0; u < VPT; ++u) e[u * NP] = acc[u];
            }
        }
        __syncthreads();
        for (int i = tid; i < erow; i += kThreads) {
            T a = ex[kHierLevels - 1][i];
            for (int k = 1; k < kTopSplit; ++k) a += ex[kHierLevels - 1][(size_t)k * erow + i];
            ex[kHierLevels - 1][i] = a;
        }
        // ---- local expansions down
        for (int l = kHierLevels - 2; l >= 0; --l) {
            __syncthreads();
            for (int it = tid; it < nloc[l] * erow; it += kThreads) {
                const int bl = it / erow, e = it % erow;
                const int q = e % NP, cv = e / NP;
                const int i = (l0 >> (2 * l)) + bl;
                const T* par = ex[l + 1] + (size_t)(nloc[l + 1] > 1 ? bl / 4 : 0) * erow + cv * NP;
                const T* w = P.tr + (l * 4 + (i & 3)) * NP * NP + q;
                T acc = ex[l][it];
#pragma unroll
                for (int p = 0; p < NP; ++p) acc += w[p * NP] * par[p];
                ex[l][it] = acc;
            }
        }
        __syncthreads();
    }
    // ---- near field, local expansions at the rows, output
    const int half = lane >> 4, r = lane & 15;
    const int gvs = NVT / NV;
    for (int item = warp; item < SL * gvs; item += kWarps) {
        const int li = item / gvs, gv = item % gvs;
        const int leaf = l0 + li;
        if (leaf >= leaves || leaf < P.leaf0) continue;
        const int v0 = gv * NV + half * KV;
        const T* xv = xs + (size_t)v0 * XS + NC * li * kHierLeaf;
        const T* hb = hw + 2 * li * kHierLeaf + r;
        T acc[KV][2][NC];
#pragma unroll
        for (int k = 0; k < KV; ++k)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[k][0][c] = acc[k][1][c] = T(0);
        // columns b0 .. b0 + NB - 1: NB x NC = 4 inputs per vector
        constexpr int NB = 4 / NC;
        // rows r + 16 meet no column below 16 (s is zero left of the diagonal)
#pragma unroll 2
        for (int b0 = 0; b0 < 2 * kHierLeaf; b0 += NB) {
            T A0[NB][NC], A1[NB][NC];
#pragma unroll
            for (int j = 0; j < NB; ++j) {
                const T s0 = sw[b0 + j - r], s1 = sw[b0 + j - r - 16];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    A0[j][c] = s0 * hb[b0 + j + c];
                    A1[j][c] = s1 * hb[b0 + j + c + 16];
                }
            }
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                T x[4];
#pragma unroll
                for (int q = 0; q < 4; q += QV) {
                    Vec16<T> t;
                    t.load(xv + (size_t)k * XS + NC * b0 + q);
#pragma unroll
                    for (int j = 0; j < QV; ++j) x[q + j] = t.v[j];
                }
#pragma unroll
                for (int j = 0; j < NB; ++j)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        acc[k][0][c] += A0[j][c] * x[j * NC + c];
                        acc[k][1][c] += A1[j][c] * x[j * NC + c];
                    }
            }
        }
        if (leaves > 2) {
            const T* e = ex[0] + (size_t)li * erow;
#pragma unroll
            for (int q = 0; q < NP; q += QV) {
                T w0[QV], w1[QV];
#pragma unroll
                for (int j = 0; j < QV; ++j) {
                    w0[j] = lw[(q + j) * kHierLeaf + r];
                    w1[j] = lw[(q + j) * kHierLeaf + r + 16];
                }
#pragma unroll
                for (int k = 0; k < KV; ++k)
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        Vec16<T> t;
                        t.load(e + (c * NVT + v0 + k) * NP + q);
#pragma unroll
                        for (int j = 0; j < QV; ++j) {
                            acc[k][0][c] += w0[j] * t.v[j];
                            acc[k][1][c] += w1[j] * t.v[j];
                        }
                    }
            }
        }
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
            const int64_t kp = (int64_t)NC * ((int64_t)leaf * kHierLeaf + r + 16 * rr);
            // packed pair -> coefficients k .. k + NC - 1 (components swapped when reversed)
            const int64_t k0 = P.rev ? P.npk - NC - kp : kp;
            T d[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const int64_t k = k0 + c;
                d[c] = (k >= 0 && k < P.n) ? P.dout[k] : T(0);
                if (P.sign_out && (k & 1)) d[c] = -d[c];
            }
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                int64_t base, len;
                vector_at<T, RAGGED>(P, g0 + v0 + k, &base, &len);
                T y[NC];
#pragma unroll
                for (int c = 0; c < NC; ++c) y[c] = acc[k][rr][P.rev ? NC - 1 - c : c] * d[c];
                if (k0 == 0 && len > 0 && P.a00) y[0] += P.a00[0] * P.in[base];
                T* o = P.out + base + k0;
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (k0 + c >= 0 && k0 + c < len) o[c] = y[c];
            }
        }
    }
}

// --------------------------------------------------------------------------- direct product
//
// Short vectors, few of them: every entry of the triangle once, no far field (one launch).  A
// CTA stages the scaled inputs and the tables in shared memory; a warp takes one packed row
// of V vectors, lanes along the columns (s from the diagonal on, h and the inputs all read with
// consecutive lanes on consecutive places).
template <typename T, int NC, int V>
__global__ void __launch_bounds__(kThreads) k_hier_direct(const __grid_constant__ HierParams<T> P,
                                                          int m, int rows) {
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
    for (int r = warp; r < rows && a0 + r < m; r += kWarps) {
        T acc[V][NC];
#pragma unroll
        for (int v = 0; v < V; ++v)
#pragma unroll
            for (int c = 0; c < NC; ++c) acc[v][c] = T(0);
        for (int b = r + lane; b < w; b += 32) {
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
        if (lane < NC * V) {
            T y = T(0);
#pragma unroll
            for (int v = 0; v < V; ++v)
#pragma unroll
                for (int c = 0; c < NC; ++c)
                    if (lane == v * NC + c) y = acc[v][c];
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

// ------------------------------------------------------------------------------ host side

// Chebyshev points of a box of `size` packed indices, rounded to distinct integers.
void hier_points(int size, int P, int* x) {
    const double pi = 3.14159265358979323846;
    for (int i = 0; i < P; ++i)
        x[i] = (int)std::lrint(0.5 * size - 0.5 -
                               0.5 * (size - 1) * std::cos(pi * (2 * i + 1) / (2.0 * P)));
    for (int i = 1; i < P; ++i) x[i] = std::max(x[i], x[i - 1] + 1);
    for (int i = P - 1; i >= 0; --i) x[i] = std::min(x[i], size - P + i);
}

double lagrange(const int* x, int P, int i, double at) {
    double v = 1.0;
    for (int j = 0; j < P; ++j)
        if (j != i) v *= (at - x[j]) / (double)(x[i] - x[j]);
    return v;
}

// table copies in execute precision: s_m = t[stride m] (32 zeros before, zero past mpad),
// hf_l = h[stride l], hr_i = hf[2 mpad - 1 - i]; entry 0 of h dropped where (0, 0) is direct
template <typename T>
__global__ void k_hier_tables(const double* __restrict__ t, const double* __restrict__ h,
                              int64_t mpad, int stride, int j0, T* __restrict__ s,
                              T* __restrict__ hf, T* __restrict__ hr) {
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i < kHierSZero) s[i - kHierSZero] = T(0);
    if (i < mpad) s[i] = (T)t[stride * i];
    if (i < 2 * mpad + kHierHPad) {
        const bool in = i < 2 * mpad;
        const T v = (!in || (j0 == 1 && i == 0)) ? T(0) : (T)h[stride * i];
        hf[i] = v;
        if (in)
            hr[2 * mpad - 1 - i] = v;
        else
            hr[i] = T(0);
    }
}

template <typename T>
int prepare_typed(Step& st, cudaStream_t s) {
    constexpr int P = HierP<T>::P;
    HierData& H = st.hier;
    const int NC = st.full ? 1 : 2;
    const int64_t m = (st.n + NC - 1) / NC;
    H.mpad = (m + kHierTop - 1) / kHierTop * kHierTop;
    // symbols of the padded length: the boxes at the end reach past n
    const int64_t N = NC * H.mpad + 2;
    double* sym = nullptr;  // t[N], h[2N-1], d1[N], d2[N]
    TDH_TRY(dev_alloc_t(&sym, (size_t)(5 * N)));
    const size_t ns = (size_t)(H.mpad + kHierSZero), nh = (size_t)(2 * H.mpad + kHierHPad);
    const size_t nw = (size_t)P * kHierLeaf + 12 * P * P;
    int rc = dev_alloc(&H.tab, sizeof(T) * (ns + 2 * nh + nw));
    if (rc == TDH_OK)
        rc = symbols_launch(st.kind, N, st.p, sym, sym + N, sym + 3 * N, sym + 4 * N, s);
    std::vector<T> w(nw);
    if (rc == TDH_OK) {
        T* tab = static_cast<T*>(H.tab);
        H.s = tab + kHierSZero;
        H.hf = tab + ns;
        H.hr = tab + ns + nh;
        H.w = tab + ns + 2 * nh;
        const int64_t cnt = 2 * H.mpad + kHierHPad;
        k_hier_tables<T><<<(unsigned)((cnt + kThreads - 1) / kThreads), kThreads, 0, s>>>(
            sym, sym + N, H.mpad, NC, (int)st.j0, static_cast<T*>(H.s), static_cast<T*>(H.hf),
            static_cast<T*>(H.hr));
        int x[kHierLevels][P];
        for (int l = 0; l < kHierLevels; ++l) hier_points(hier_size(l), P, x[l]);
        for (int p = 0; p < P; ++p)
            for (int a = 0; a < kHierLeaf; ++a)
                w[(size_t)p * kHierLeaf + a] = (T)lagrange(x[0], P, p, a);
        for (int l = 1; l < kHierLevels; ++l)
            for (int c = 0; c < 4; ++c)
                for (int p = 0; p < P; ++p)
                    for (int q = 0; q < P; ++q)
                        w[(size_t)P * kHierLeaf + (((l - 1) * 4 + c) * P + p) * P + q] =
                            (T)lagrange(x[l], P, p, c * hier_size(l - 1) + x[l - 1][q]);
        cudaError_t e = cudaGetLastError();
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(H.w, w.data(), sizeof(T) * nw, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            set_error("hierarchical tables: %s", cudaGetErrorString(e));
            rc = TDH_ERR_CUDA;
        }
    }
    dev_free(sym);
    if (rc == TDH_OK) H.on = H.use = 1;
    H.use_ragged = H.use && NC == 2;
    return rc;
}

// Launch shape of one execute.
struct Shape {
    int NV;           // vectors per warp of the down kernel
    int gv, gu;       // warp groups of vectors per CTA (down, up)
    int seg_leaves;
    int64_t chunk;    // vectors per pass over the moment scratch
};

template <typename T>
size_t down_smem(int NC, int SL, int NVT) {
    constexpr int P = HierP<T>::P;
    size_t e = (size_t)NVT * (NC * (SL + 1) * kHierLeaf + 16 / sizeof(T));
    e += kHierSZero + 8 * kHierLeaf + 2 * SL * kHierLeaf + 10 * kHierLeaf + P * kHierLeaf;
    size_t boxes = kTopSplit;
    for (int l = 0; l < kHierLevels - 1; ++l) boxes += std::max(1, SL >> (2 * l));
    return sizeof(T) * (e + boxes * NC * NVT * P);
}

template <typename T>
size_t up_smem(int NC, int NVT) {
    constexpr int P = HierP<T>::P;
    constexpr int VW = 32 / P;
    return sizeof(T) * ((size_t)kWarps * VW * (NC * kHierLeaf + 16 / sizeof(T)) +
                        (size_t)(kHierTopLeaves + kHierTopLeaves / 4 + kHierTopLeaves / 16) * NC *
                            NVT * P);
}

constexpr size_t kMaxSmem = 227 * 1024;

template <typename T>
Shape choose_shape(int NC, int64_t leaves, int64_t batch) {
    Shape sh{};
    const int vmax = sizeof(T) == 4 ? 16 : 8;
    sh.NV = batch >= vmax * 3 / 4 ? vmax : (batch > 2 ? 8 : 2);
    const int64_t groups = (batch + sh.NV - 1) / sh.NV;
    // the longest segments that still give every SM a few CTAs
    const int64_t want = 4 * (int64_t)sm_count();
    sh.seg_leaves = 16;
    while (sh.seg_leaves > 1 &&
           (sh.seg_leaves >= 4 * leaves || (leaves / sh.seg_leaves) * groups < want))
        sh.seg_leaves /= 4;
    // short segments: several vector groups per CTA, so that all eight warps have a leaf
    sh.gv = 1;
    const int64_t per = std::min<int64_t>(leaves, sh.seg_leaves);
    while (per * sh.gv < kWarps && (int64_t)(2 * sh.gv) * want <= groups * ((leaves + per - 1) / per))
        sh.gv *= 2;
    while (sh.gv > 1 && down_smem<T>(NC, sh.seg_leaves, sh.NV * sh.gv) > kMaxSmem) sh.gv /= 2;
    sh.gu = 1;
    return sh;
}

template <typename T>
cudaError_t launch_cfg(void (*kern)(const HierParams<T>), unsigned grid, size_t smem,
                       cudaStream_t s, bool pdl, const HierParams<T>& P) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kThreads);
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
    auto kern = k_hier_up<T, NC, RAGGED>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem);
    });
    if (e == cudaSuccess) e = launch_cfg<T>(kern, grid, up_smem<T>(NC, P.unvt), s, false, P);
    if (e != cudaSuccess) {
        set_error("hierarchical moments: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, int NV, bool RAGGED>
int launch_down_nv(const HierParams<T>& P, unsigned grid, bool pdl, cudaStream_t s) {
    auto kern = k_hier_down<T, NC, NV, RAGGED>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem - 1024);
    });
    if (e == cudaSuccess)
        e = launch_cfg<T>(kern, grid, down_smem<T>(NC, P.seg_leaves, P.nvt), s, pdl, P);
    if (e != cudaSuccess) {
        set_error("hierarchical product: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, bool RAGGED>
int launch_down(const HierParams<T>& P, int NV, unsigned grid, bool pdl, cudaStream_t s) {
    if constexpr (sizeof(T) == 4)
        if (NV == 16) return launch_down_nv<T, NC, 16, RAGGED>(P, grid, pdl, s);
    if (NV == 8) return launch_down_nv<T, NC, 8, RAGGED>(P, grid, pdl, s);
    return launch_down_nv<T, NC, 2, RAGGED>(P, grid, pdl, s);
}

// The direct product's shared memory, and whether it is the faster way: its work is m^2 B
// multiply-adds, that of the tree a few launches and some hundred operations per coefficient.
template <typename T>
size_t direct_smem(int NC, int64_t m, int rows, int V) {
    return sizeof(T) * (size_t)(2 * m + rows + 1 + V * NC * m);
}
template <typename T>
bool direct_serves(int NC, int64_t m, int64_t batch) {
    const double work = (double)m * (double)m * (double)batch * NC;
    return m <= 4096 && work <= (sizeof(T) == 4 ? 1 << 24 : 1 << 20);
}

template <typename T, int NC, int V>
int launch_direct(const HierParams<T>& P, int64_t m, cudaStream_t s) {
    auto kern = k_hier_direct<T, NC, V>;
    static PerDevice once;
    cudaError_t e = per_device(once, [&](int*) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)kMaxSmem);
    });
    const int rows = kWarps;
    const int64_t grid = (m + rows - 1) / rows * ((P.batch + V - 1) / V);
    if (e == cudaSuccess) {
        kern<<<(unsigned)grid, kThreads, direct_smem<T>(NC, m, rows, V), s>>>(P, (int)m, rows);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("direct product: %s", cudaGetErrorString(e));
        return TDH_ERR_CUDA;
    }
    note_launches(1);
    return TDH_OK;
}

template <typename T, int NC, bool RAGGED>
int run_typed(const Step& st, const void* in, void* out, const int64_t* offs, int64_t batch,
              int adjoint, const int* list, const int* count, cudaStream_t s) {
    constexpr int NP = HierP<T>::P;
    const HierData& H = st.hier;
    const int64_t m = (st.n + NC - 1) / NC;
    HierParams<T> P{};
    P.n = st.n;
    P.npk = NC * H.mpad;
    P.s = static_cast<const T*>(H.s);
    // reversed: packed index a' + b' meets hf[2 (mpad - 1) - a' - b' (+ 1 in channel 0)]
    P.hh = static_cast<const T*>(adjoint ? H.hr : H.hf) + (adjoint && NC == 1 ? 1 : 0);
    P.lw = static_cast<const T*>(H.w);
    P.tr = P.lw + NP * kHierLeaf;
    P.din = static_cast<const T*>(adjoint ? st.d1x : st.d2x);
    P.dout = static_cast<const T*>(adjoint ? st.d2x : st.d1x);
    P.a00 = st.j0 == 1 ? static_cast<const T*>(st.row0) : nullptr;
    P.rev = adjoint;
    P.sign_in = st.sign_in;
    P.sign_out = st.sign_out;
    if (adjoint) {
        P.leaf0 = (int)((H.mpad - m) / kHierLeaf);
        P.leaves = (int)(H.mpad / kHierLeaf);
    } else {
        P.leaf0 = 0;
        P.leaves = (int)((m + kHierLeaf - 1) / kHierLeaf);
    }
    for (int l = 0; l < kHierLevels; ++l) {
        int x[NP];
        hier_points(hier_size(l), NP, x);
        for (int p = 0; p < NP; ++p) P.x[l][p] = (short)x[p];
    }
    const int64_t real_leaves = (m + kHierLeaf - 1) / kHierLeaf;
    if (!RAGGED && direct_serves<T>(NC, m, batch)) {
        P.batch = batch;
        P.in = static_cast<const T*>(in);
        P.out = static_cast<T*>(out);
        return batch == 1 ? launch_direct<T, NC, 1>(P, m, s) : launch_direct<T, NC, 4>(P, m, s);
    }
    const Shape sh = choose_shape<T>(NC, real_leaves, batch);
    P.seg_leaves = sh.seg_leaves;
    P.nvt = sh.NV * sh.gv;
    P.unvt = 32 / NP;
    P.nseg = (P.leaves + sh.seg_leaves - 1) / sh.seg_leaves;
    const int64_t ntop = (P.leaves + kHierTopLeaves - 1) / kHierTopLeaves;
    // moments of every box of a vector; at most about 1 GB of them at a time
    int64_t boxes[kHierLevels], total = 0;
    for (int l = 0; l < kHierLevels; ++l) total += boxes[l] = (H.mpad / kHierLeaf) >> (2 * l);
    const bool far = real_leaves > 2;
    const int64_t per_vec = total * NC * NP * (int64_t)sizeof(T);
    int64_t chunk = std::max<int64_t>(1, ((int64_t)1 << 30) / per_vec);
    chunk = std::min(chunk, (int64_t)INT32_MAX / 2 / std::max<int64_t>(P.nseg, ntop));
    const int unit = std::max(P.nvt, P.unvt);  // both powers of two
    chunk = std::max<int64_t>(unit, chunk / unit * unit);
    chunk = std::min<int64_t>(chunk, (batch + unit - 1) / unit * unit);
    T* mom = nullptr;
    if (far) TDH_TRY(scratch_alloc(reinterpret_cast<void**>(&mom), (size_t)(per_vec * chunk), s));
    P.bpad = chunk;
    for (int l = 0; l < kHierLevels; ++l) {
        P.mom[l] = mom;
        if (mom) mom += boxes[l] * NC * NP * chunk;
    }
    int rc = TDH_OK;
    for (int64_t b0 = 0; rc == TDH_OK && b0 < batch; b0 += chunk) {
        const int64_t nb = std::min(chunk, batch - b0);
        P.batch = nb;
        P.in = static_cast<const T*>(in);
        P.out = static_cast<T*>(out);
        if constexpr (RAGGED) {
            P.offs = offs;
            P.list = list + b0;
            P.first = b0;
            P.count = count;
        } else {
            P.in += b0 * st.n;
            P.out += b0 * st.n;
        }
        if (far) {
            const int64_t gu = ((nb + P.nvt - 1) / P.nvt * P.nvt + P.unvt - 1) / P.unvt;
            rc = launch_up<T, NC, RAGGED>(P, (unsigned)(gu * ntop), s);
        }
        if (rc == TDH_OK)
            rc = launch_down<T, NC, RAGGED>(
                P, sh.NV, (unsigned)((nb + P.nvt - 1) / P.nvt * P.nseg), far, s);
    }
    if (far) scratch_free(P.mom[0], s);
    return rc;
}

template <typename T>
int ragged_typed(const Step& st, const void* in, void* out, const int64_t* offs, int64_t batch,
                 cudaStream_t s) {
    const int unit = 2 * kHierLeaf;
    const int bins = (int)((st.n + unit - 1) / unit);
    int* scr = nullptr;  // hist[bins + 1], list[batch]
    TDH_TRY(scratch_alloc(reinterpret_cast<void**>(&scr), sizeof(int) * (size_t)(bins + 1 + batch), s));
    int* list = scr + bins + 1;
    int rc = TDH_OK;
    cudaError_t e = cudaMemsetAsync(scr, 0, sizeof(int) * (size_t)(bins + 1), s);
    const unsigned grid = (unsigned)((batch + kThreads - 1) / kThreads);
    const char* ci = static_cast<const char*>(in);
    const char* co = static_cast<const char*>(out);
    if (e == cudaSuccess) {
        k_hier_hist<<<grid, kThreads, 0, s>>>(offs, batch, st.n, unit, bins, scr, ci, co,
                                              (int)sizeof(T), st.status);
        k_hier_scan<<<1, kSortThreads, 0, s>>>(scr, bins);
        k_hier_scatter<<<grid, kThreads, 0, s>>>(offs, batch, st.n, unit, bins, scr, list, ci, co,
                                                 (int)sizeof(T));
        note_launches(3);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        set_error("ragged lists: %s", cudaGetErrorString(e));
        rc = TDH_ERR_CUDA;
    }
    if (rc == TDH_OK)
        rc = run_typed<T, 2, true>(st, in, out, offs, batch, 0, list, scr + bins, s);
    scratch_free(scr, s);
    return rc;
}

}  // namespace

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
        return st.full ? run_typed<float, 1, false>(st, in, out, nullptr, batch, adjoint, nullptr,
                                                    nullptr, s)
                       : run_typed<float, 2, false>(st, in, out, nullptr, batch, adjoint, nullptr,
                                                    nullptr, s);
    return st.full ? run_typed<double, 1, false>(st, in, out, nullptr, batch, adjoint, nullptr,
                                                 nullptr, s)
                   : run_typed<double, 2, false>(st, in, out, nullptr, batch, adjoint, nullptr,
                                                 nullptr, s);
}

int hier_launch_ragged(const Step& st, int prec, const void* in, void* out, const int64_t* offs,
                       int64_t batch, cudaStream_t s) {
    return prec != TDH_FP64 ? ragged_typed<float>(st, in, out, offs, batch, s)
                            : ragged_typed<double>(st, in, out, offs, batch, s);
}

}  // namespace tdh
