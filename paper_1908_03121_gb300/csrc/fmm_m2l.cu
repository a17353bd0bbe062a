// Same-level pass (Sec. 4.3, second step; Sec. 5.1 moves it to the GPU).
//
// Every cell A gathers, from each same-level source B that the opening rule
// selects, the order-3 Taylor coefficients of B's potential at A's centre of
// mass, in level units (lengths in cell widths, G factored out):
//   L^(n)_A -= sum_{m: n+m<=3} ((-1)^m / m!) M_B^(m) . D^(n+m)(R),
//   R = X_A - X_B,
// and the angular-momentum correction
//   dL1_A,i += (1/6) sum_jkl D4_ijkl(R) [M3_B - (M0_B / M0_A) M3_A]_jkl.
// Sec. 4.3 lists four kinds by node refinement; this file has one kernel per
// kind of target, as the paper's GPU port fuses multipole<-multipole with
// multipole<-monopole:
//   mp_kernel    refined targets: multipole<-multipole (well-separated
//                sources) and multipole<-monopole (all candidate leaf
//                sources) -- the "455 flop" kernel of Sec. 4.3; in the mixed
//                precision also mp_split_kernel (trees with few sub-grids)
//                and mp2_kernel (two targets per thread, a tuning), in the
//                wide element types mpw_kernel (fmm_wide.cuh's algebra);
//   mono_kernel  leaf targets, leaf sources: monopole<-monopole, a 1-in,
//                4-out convolution whose per-offset weights are tabulated
//                (wide types: mono_wide_kernel in fmm_mono_wide.cuh);
//   mx_kernel    leaf targets next to refined nodes: monopole<-multipole;
//   root_kernel  the single node of level 1 of each tree (all pairs are
//                candidates there); wide types: rootw_kernel.
// Design (GB300-first, unlike the paper's 8x64-thread launches per node fed
// from 128 streams): persistent CTAs pull whole sub-grids from cost-sorted
// work queues; a warp holds 32 targets of one child parity so the stencil
// loop is warp-uniform; leaf-source masses of the 26-neighbour halo are staged
// once per sub-grid into a parity-split, bank-padded shared-memory window;
// refined-source moments stream through L1 as four vector loads from a
// parity-split packed layout, so a warp's loads are contiguous.  Orders 2-4
// of the derivative tensors are traceless, so the contraction works in
// traceless bases (fmm_tensor.cuh): 16 accumulated components instead of 20,
// 16 packed source values instead of 20, and about a quarter fewer products.
// Mixed precision: offsets are formed from double-precision centres of mass
// (packed as offsets from the cell centre, in cell widths), the contraction
// runs in float with per-chunk sums folded into (hi, lo) pairs by TwoSum, and
// the correction's compensated sum is stored and carried down in double.
// Wide element types (double, and dfloat: pairs of floats, fmm_dfloat.cuh, the
// conserving precision): both are bound by their arithmetic pipe, so their
// kernels are written for the fewest operations (fmm_wide.cuh); dfloat
// evaluates offsets, contraction and sums in double-float, so each pair's
// contributions to A and to B cancel in momentum and angular momentum to about
// 1e-13, as in FP64.
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "fmm_convert.cuh"
#include "fmm_internal.h"
#include "fmm_tensor.cuh"
#include "fmm_wide.cuh"

namespace fmm {

namespace {

// element types of the three precisions: float (mixed), dfloat (conserving),
// double (FP64)
template <typename T> constexpr bool kF32 = std::is_same<T, float>::value;
template <typename T> constexpr bool kDF = std::is_same<T, dfloat>::value;

template <typename T>
__device__ __forceinline__ T ldg_t(const T *p)
{
    if constexpr (kDF<T>) {
        const float2 f = __ldg(reinterpret_cast<const float2 *>(p));
        return dfloat(f.x, f.y);
    } else {
        return __ldg(p);
    }
}

constexpr int kThreads = 256;   // 8 warps = the 8 child parities
constexpr int kChunk = 16;      // stencil entries per compensated chunk
constexpr int Q_MP = 0, Q_MONO = 1, Q_MX = 2;   // work-queue heads (Q_MX: the fused launch)

struct KParams {
    const NodeInfo *info;
    const int32_t *nbr;
    const int32_t *list;
    int32_t n_items;
    int32_t *counter;
    const float4 *stencil_f;  // stencil entries: offsets as floats, window offset's bits in w
    const float *coef;       // monopole weights of parity 0 (mixed)
    const int32_t *mono_woff;  // [8][ent_stride] window offsets in parity 0's order, reflected
    const uint16_t *mono_woff16;  // the same, in bytes
    int n_far, n_near;       // identical for every parity
    int ent_stride;          // entries reserved per parity
    const int4 *mx_targets;  // monopole<-multipole targets (node, cell, warp's pair base, count)
    int32_t n_mx;            // monopole<-multipole targets the multipole launch takes (0: none)
    int32_t *mx_counter;     // their queue head
    const int2 *mx_pairs;    // (packed-moment offset, stencil entry); pair k of target
                             // 32 w + j at its warp's base + 32 k + j
    int reach, py, pz, sub_stride;
    const void *mass;
    const void *mp;
    int mp_limit;            // elements of mp: decoded window offsets below it only; the
                             // row starting there holds zeros
    void *L;
    float *Lc;
    double *dL1;
    int far_o2;              // cells at squared offset >= far_o2 are well separated
};

// ------------------------------------------------------------------ pack
// a double as the element type (double-float: split with the conversions on
// the integer pipe)
template <typename T>
__device__ __forceinline__ T elem_from_double(double v)
{
    if constexpr (kDF<T>) return df_from_double(v);
    else return T(v);
}

// Mixed precision: everything but the centre-of-mass offset in float, with
// the double -> float conversions on the integer pipe (GB300's FP64 unit,
// which also runs conversions, would otherwise bound this pass); the
// moments' float rounding is the contraction's own precision.
// (the FP64 moments are read once, with the evict-first hint, so that they
// do not push the packed values just written out of L2, where the
// multipole kernel reads them next)
__device__ __forceinline__ void pack_float(const NodeInfo &ni, const double *__restrict__ levels,
                                           const double *__restrict__ Mn,
                                           const double *__restrict__ comc, int x, int y, int z,
                                           int pi, float *__restrict__ mass_node,
                                           float *__restrict__ mp, double lo_x, double lo_y,
                                           double lo_z)
{
    mass_node[pi] = d2f_rn(__ldcs(Mn));
    if (ni.mp_row < 0) return;
    const double h = levels[ni.level * LEVEL_FIELDS + LV_H];
    const float ih = d2f_rn(levels[ni.level * LEVEL_FIELDS + LV_IH]);
    const double ctr[3] = {lo_x + (8.0 * ni.ix + x + 0.5) * h, lo_y + (8.0 * ni.iy + y + 0.5) * h,
                           lo_z + (8.0 * ni.iz + z + 0.5) * h};
    float d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = d2f_rn(__ldcs(comc + a * NCELL) - ctr[a]) * ih;
    const float w2 = 0.5f * ih * ih, w3 = (1.0f / 6.0f) * ih * ih * ih;
    float A2[6], A3[10];
#pragma unroll
    for (int q = 0; q < 6; ++q) A2[q] = d2f_rn(__ldcs(Mn + (4 + q) * NCELL)) * (float(mult2(q)) * w2);
#pragma unroll
    for (int q = 0; q < 10; ++q) A3[q] = d2f_rn(__ldcs(Mn + (10 + q) * NCELL)) * (float(mult3(q)) * w3);
    const float v[16] = {d[0],          d[1],          d[2],          mass_node[pi],
                         A2[0] - A2[5], A2[3] - A2[5], A2[1],         A2[2],
                         A2[4],         A3[0] - A3[5], A3[1] - A3[8], A3[2] - A3[9],
                         A3[3] - A3[5], A3[4],         A3[6] - A3[8], A3[7] - A3[9]};
    float4 *out = reinterpret_cast<float4 *>(mp + (size_t(ni.mp_row) * 4 * NCELL + pi) * 4);
#pragma unroll
    for (int g = 0; g < 4; ++g)
        out[size_t(g) * NCELL] = make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
}

// mass[node][pi] = M0 for every node.  Refined nodes also get, in level
// units, four groups of four values at mp[row][g][pi][0..3]:
//   g0 = (delta, M0), delta = (X - centre) / h (first, so that its x and y
//        land in an aligned register pair for the paired FP32 subtraction),
//   g1 = B2[0..3], g2 = (B2[4], B3[0..2]), g3 = B3[3..6],
// float: the traceless projections of A2 = mult M2 / (2 h^2),
// A3 = mult M3 / (6 h^3); double-float and double: the traceless parts
// themselves, t2 = (3/2) T2 / h^2 (xx yy xy xz yz) and t3 = (5/2) T3 / h^3 (xxx
// xxy xxz xyy xyz yyy yyz), see fmm_wide.cuh.
template <typename T>
__global__ void __launch_bounds__(512) pack_kernel(const NodeInfo *__restrict__ info,
                                                   const int32_t *__restrict__ nodes,
                                                   const double *__restrict__ levels,
                                                   const double *__restrict__ M,
                                                   const double *__restrict__ com,
                                                   T *__restrict__ mass, T *__restrict__ mp,
                                                   double lo_x, double lo_y, double lo_z)
{
    const int node = nodes ? nodes[blockIdx.x] : int(blockIdx.x);   // a list, or every node
    const NodeInfo ni = info[node];
    const int c = threadIdx.x;
    const int x = c & 7, y = (c >> 3) & 7, z = c >> 6;
    const int pi = parity_index(x, y, z);
    const double *Mn = M + size_t(node) * NCOMP * NCELL + c;
    if constexpr (kF32<T>) {
        pack_float(ni, levels, Mn, com + size_t(node) * 3 * NCELL + c, x, y, z, pi, mass + size_t(node) * NCELL,
                   mp, lo_x, lo_y, lo_z);
        return;
    }
    mass[size_t(node) * NCELL + pi] = elem_from_double<T>(Mn[0]);
    if (ni.mp_row < 0) return;
    const double h = levels[ni.level * LEVEL_FIELDS + LV_H];
    const double ih = levels[ni.level * LEVEL_FIELDS + LV_IH];
    const double ctr[3] = {lo_x + (8.0 * ni.ix + x + 0.5) * h, lo_y + (8.0 * ni.iy + y + 0.5) * h,
                           lo_z + (8.0 * ni.iz + z + 0.5) * h};
    double d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = (com[(size_t(node) * 3 + a) * NCELL + c] - ctr[a]) * ih;
    // traceless parts: T2 = M2 - delta tr/3, T3 = M3 - (delta v, three terms)/5
    // with v_k = M3_iik; symmetric order M2 xx xy xz yy yz zz, M3 xxx xxy xxz
    // xyy xyz xzz yyy yyz yzz zzz
    const double w2 = 1.5 * ih * ih, w3 = 2.5 * ih * ih * ih;
    double m2[6], m3[10];
#pragma unroll
    for (int q = 0; q < 6; ++q) m2[q] = Mn[(4 + q) * NCELL];
#pragma unroll
    for (int q = 0; q < 10; ++q) m3[q] = Mn[(10 + q) * NCELL];
    const double tr = (m2[0] + m2[3] + m2[5]) * (1.0 / 3.0);
    const double vx = 0.2 * (m3[0] + m3[3] + m3[5]), vy = 0.2 * (m3[1] + m3[6] + m3[8]),
                 vz = 0.2 * (m3[2] + m3[7] + m3[9]);
    const double v[16] = {d[0],
                          d[1],
                          d[2],
                          Mn[0],
                          w2 * (m2[0] - tr),
                          w2 * (m2[3] - tr),
                          w2 * m2[1],
                          w2 * m2[2],
                          w2 * m2[4],
                          w3 * (m3[0] - 3.0 * vx),
                          w3 * (m3[1] - vy),
                          w3 * (m3[2] - vz),
                          w3 * (m3[3] - vx),
                          w3 * m3[4],
                          w3 * (m3[6] - 3.0 * vy),
                          w3 * (m3[7] - vz)};
    T *out = mp + (size_t(ni.mp_row) * 4 * NCELL + pi) * 4;
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
        for (int j = 0; j < 4; ++j) out[size_t(g) * NCELL * 4 + j] = elem_from_double<T>(v[4 * g + j]);
}

// ------------------------------------------------------------ common bits
__device__ __forceinline__ int pull_item(int32_t *counter, int *s_item)
{
    if (threadIdx.x == 0) *s_item = atomicAdd(counter, 1);
    __syncthreads();
    return *s_item;
}

// Stage the halo window of leaf-cell masses around a target node: window
// cell u in [0, 8 + 2R)^3 holds the source at node-local position u - R, or 0
// when that source is refined or absent.  Layout: parity sub-window
// q = (ux&1) + 2(uy&1) + 4(uz&1), then (ux>>1) + py (uy>>1) + pz (uz>>1).
// One (ux, uy) column per thread pass, z innermost; the parity index and the
// window address both split into an (x, y) part and a z part.  The copies go
// through cp.async (global -> shared without registers; sources that are
// refined or absent are zero-filled by a zero source size), so every load of
// the window is in flight at once.  The caller commits and waits.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst, const T *src, bool valid)
{
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "cp.async element size");
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src),
                 "n"(int(sizeof(T))), "r"(valid ? int(sizeof(T)) : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }
// all but the newest N groups
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
// 16 bytes, zeros if not valid
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid)
{
    const unsigned d = unsigned(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 16 : 0)
                 : "memory");
}

// With s_row given (the multipole-target kernel), a refined source's cell
// holds instead the offset of its packed moments (row and parity index),
// encoded by window_index as a value with the sign bit set (masses are not
// negative); without, it holds 0.  The kernels use a decoded offset only
// below mp_limit, so an invalid negative density can give wrong results but
// no access outside the packed moments.
template <typename T>
__device__ __forceinline__ T window_index(int idx)
{
    if constexpr (kF32<T>) {
        return __int_as_float(-1 - idx);
    } else if constexpr (kDF<T>) {
        return dfloat(__int_as_float(-1 - idx), 0.f);
    } else {
        return __longlong_as_double(-1ll - idx);
    }
}

// whether a window value is a refined source's moment offset below limit,
// and that offset: -1 - bits is the offset for a refined source and
// negative (a large unsigned value) for a mass, whose bits are not
// negative, so one unsigned comparison tells both apart and bounds the
// offset
template <typename T>
__device__ __forceinline__ bool window_moments(T v, int limit, int &idx)
{
    if constexpr (kF32<T>) {
        const unsigned u = unsigned(-1 - __float_as_int(v));
        idx = int(u);
        return u < unsigned(limit);
    } else if constexpr (kDF<T>) {
        const unsigned u = unsigned(-1 - __float_as_int(v.hi));
        idx = int(u);
        return u < unsigned(limit);
    } else {
        const unsigned long long u = static_cast<unsigned long long>(-1ll - __double_as_longlong(v));
        idx = int(u);
        return u < static_cast<unsigned long long>(limit);
    }
}

// whether a window value encodes a refined source (sign bit set)
template <typename T>
__device__ __forceinline__ bool window_refined(T v)
{
    if constexpr (kF32<T>) {
        return __float_as_int(v) < 0;
    } else if constexpr (kDF<T>) {
        return __float_as_int(v.hi) < 0;
    } else {
        return __double_as_longlong(v) < 0;
    }
}

// Window geometry of reach R: the host's pitches (same pad_to), as
// compile-time constants; RR = 0 takes them from the kernel parameters.
template <int RR>
struct WinGeo {
    static constexpr int R = RR, SUB = 4 + RR, E = 8 + 2 * RR;
    static constexpr int PY = pad_to(SUB, 12), PZ = pad_to(SUB * PY, 16), SUB_STRIDE = SUB * PZ;
};

template <typename T, int RR = 0>
__device__ __forceinline__ void stage_window_async(T *W, const int *s_nbr, const int *s_leaf,
                                                   const T *__restrict__ mass, const KParams &P,
                                                   const int *s_row = nullptr)
{
    using G = WinGeo<RR>;
    const int R = RR ? G::R : P.reach;
    const int E = RR ? G::E : 8 + 2 * R;
    const int py = RR ? G::PY : P.py, pz = RR ? G::PZ : P.pz;
    const int sub_stride = RR ? G::SUB_STRIDE : P.sub_stride;
    for (int t = threadIdx.x; t < E * E; t += blockDim.x) {
        const int ux = t % E, uy = t / E;
        const int bx = ux - R + 8, by = uy - R + 8;           // >= 1
        const int sxy = (bx >> 3) + 3 * (by >> 3);
        const int lx = bx & 7, ly = by & 7;
        const int pxy = ((lx & 1) + 2 * (ly & 1)) * 64 + (lx >> 1) + 4 * (ly >> 1);
        const int wxy = ((ux & 1) + 2 * (uy & 1)) * sub_stride + (ux >> 1) + py * (uy >> 1);
#pragma unroll 4
        for (int uz = 0; uz < E; ++uz) {
            const int bz = uz - R + 8;
            const int slot = sxy + 9 * (bz >> 3);
            const int lz = bz & 7;
            const bool ok = s_leaf[slot] != 0;
            const int pi = pxy + 256 * (lz & 1) + 16 * (lz >> 1);
            const T *src = ok ? mass + size_t(s_nbr[slot]) * NCELL + pi : mass;
            const int wi = wxy + 4 * (uz & 1) * sub_stride + pz * (uz >> 1);
            const int row = s_row ? s_row[slot] : -1;
            if (row >= 0)
                W[wi] = window_index<T>((row * 4 * NCELL + pi) * 4);
            else
                cp_async_elem<T>(W + wi, src, ok);
        }
    }
}

// neighbour tables of the current target node into shared memory; returns,
// in threads 0-26, whether that thread's neighbour is a leaf (0 elsewhere)
__device__ __forceinline__ int load_slots(int node, const KParams &P, int *s_nbr, int *s_leaf,
                                          int *s_row)
{
    int is_leaf = 0;
    if (threadIdx.x < 27) {
        const int nb = P.nbr[node * 27 + threadIdx.x];
        s_nbr[threadIdx.x] = nb;
        int leaf = 0, row = -1;
        if (nb >= 0) {
            const NodeInfo ni = P.info[nb];
            leaf = ni.leaf_row >= 0;
            row = ni.mp_row;
        }
        s_leaf[threadIdx.x] = leaf;
        s_row[threadIdx.x] = row;
        is_leaf = leaf;
    }
    return is_leaf;
}

// a window value that is a nonzero mass or a moment offset (an absent
// source's cell holds 0 and contributes nothing)
template <typename T>
__device__ __forceinline__ bool window_nonzero(T v)
{
    if constexpr (kDF<T>) {
        return v.hi != 0.f;
    } else {
        return v != T(0);
    }
}

// Compensated accumulator: float partial sums per chunk, folded into a
// (hi, lo) pair by TwoSum.
template <int N>
struct Acc {
    float part[N];
    float hi[N];
    float lo[N];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int k = 0; k < N; ++k) part[k] = hi[k] = lo[k] = 0.f;
    }
    __device__ __forceinline__ void flush()
    {
#pragma unroll
        for (int k = 0; k < N; ++k) {
            float s, e;
            two_sum(hi[k], part[k], s, e);
            hi[k] = s;
            lo[k] += e;
            part[k] = 0.f;
        }
    }
};

// the (hi, lo) value of accumulator k
template <int N>
__device__ __forceinline__ float acc_hi(const Acc<N> &a, int k) { return a.hi[k]; }
template <int N>
__device__ __forceinline__ float acc_lo(const Acc<N> &a, int k) { return a.lo[k]; }

// Float accumulator whose (hi, lo) pairs live in shared memory, in this
// thread's column of a [components][2][threads] array: only the chunk sums
// take registers.  The first NC components are compensated; the others
// (the multipole target's orders 2-3, which reach the forces only through
// the downward shifts, scaled by the small child offsets) are plain float
// sums in registers.  Fewer pairs leave more of the SM's shared memory to
// L1, where the multipole kernel rereads the sources' packed moments.
template <int N, int NC = N, int THREADS = kThreads>
struct SmemAcc {
    float part[N];
    float *col;                       // the (hi, lo) pairs of component k < NC at col[k * 2 * THREADS]
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int k = 0; k < N; ++k) part[k] = 0.f;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            col[k * 2 * THREADS] = 0.f;
            col[(k * 2 + 1) * THREADS] = 0.f;
        }
    }
    __device__ __forceinline__ void flush()
    {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
            float s, e;
            two_sum(col[k * 2 * THREADS], part[k], s, e);
            col[k * 2 * THREADS] = s;
            col[(k * 2 + 1) * THREADS] += e;
            part[k] = 0.f;
        }
    }
};
template <int N, int NC, int THREADS>
__device__ __forceinline__ float acc_hi(const SmemAcc<N, NC, THREADS> &a, int k)
{
    return k < NC ? a.col[k * 2 * THREADS] : a.part[k];
}
template <int N, int NC, int THREADS>
__device__ __forceinline__ float acc_lo(const SmemAcc<N, NC, THREADS> &a, int k)
{
    return k < NC ? a.col[(k * 2 + 1) * THREADS] : 0.f;
}

// (the multipole kernel keeps shared-memory pairs for orders 0-1 and the correction)
constexpr int kMpPairs = 4 + 3;      // compensated float components of mp_kernel

// store component k of a target cell: level units; (hi, lo) float pairs for
// float (renormalised) and double-float (lo is zero there), else double
// Same-level results are stored with the evict-first (streaming) hint: they
// are read once, much later, by the downward pass, and left in L2 they would
// push out the packed source moments that the multipole kernel rereads.
template <typename T, class Params>
__device__ __forceinline__ void store_L(const Params &P, int node, int k, int cell, T hi, T lo)
{
    const size_t idx = (size_t(node) * NCOMP + k) * NCELL + cell;
    if constexpr (kF32<T>) {
        // renormalise so that |lo| <= ulp(hi)/2
        float s = hi + lo;
        float e = lo - (s - hi);
        __stcs(static_cast<float *>(P.L) + idx, s);
        __stcs(P.Lc + idx, e);
    } else if constexpr (kDF<T>) {
        __stcs(static_cast<float *>(P.L) + idx, hi.hi);
        __stcs(P.Lc + idx, hi.lo);
    } else {
        __stcs(static_cast<double *>(P.L) + idx, hi);
    }
}

// store -(a + b) for a traceless-dependent component
template <typename T>
__device__ __forceinline__ void store_neg_sum(const KParams &P, int node, int k, int cell,
                                              const T hi[16], const T lo[16], int a, int b)
{
    if constexpr (kF32<T>) {
        float s, e;
        two_sum(hi[a], hi[b], s, e);
        store_L<T>(P, node, k, cell, -s, -(lo[a] + lo[b] + e));
    } else {
        store_L<T>(P, node, k, cell, -(hi[a] + hi[b]), T(0));
    }
}

// the 16 traceless values of a multipole target -> 20 stored components
// values: 0 L0 | 1-3 L1 | 4-8 L2 (xx yy xy xz yz) | 9-15 L3 (xxx xxy
// xxz xyy xyz yyy yyz)
template <typename T>
__device__ __forceinline__ void store_target_values(const KParams &P, int node, int cell,
                                                    const T hi[16], const T lo[16])
{
    constexpr int direct[16] = {0, 1, 2, 3, 4, 7, 5, 6, 8, 10, 11, 12, 13, 14, 16, 17};
#pragma unroll
    for (int k = 0; k < 16; ++k) store_L<T>(P, node, direct[k], cell, hi[k], lo[k]);
    store_neg_sum<T>(P, node, 9, cell, hi, lo, 4, 5);      // zz  = -(xx + yy)
    store_neg_sum<T>(P, node, 15, cell, hi, lo, 9, 12);    // xzz = -(xxx + xyy)
    store_neg_sum<T>(P, node, 18, cell, hi, lo, 10, 14);   // yzz = -(xxy + yyy)
    store_neg_sum<T>(P, node, 19, cell, hi, lo, 11, 15);   // zzz = -(xxz + yyz)
}

template <class LA>
__device__ __forceinline__ void store_target(const KParams &P, int node, int cell, const LA &L)
{
    float hi[16], lo[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        hi[k] = acc_hi(L, k);
        lo[k] = acc_lo(L, k);
    }
    store_target_values<float>(P, node, cell, hi, lo);
}

// four consecutive values from shared memory
template <typename T>
__device__ __forceinline__ void load4_shared(const T *p, T v[4])
{
    if constexpr (kDF<T>) {
        const float4 a = reinterpret_cast<const float4 *>(p)[0];
        const float4 b = reinterpret_cast<const float4 *>(p)[1];
        v[0] = dfloat(a.x, a.y); v[1] = dfloat(a.z, a.w);
        v[2] = dfloat(b.x, b.y); v[3] = dfloat(b.z, b.w);
    } else {
        const double2 a = reinterpret_cast<const double2 *>(p)[0];
        const double2 b = reinterpret_cast<const double2 *>(p)[1];
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
}

}  // namespace
}  // namespace fmm

#include "fmm_mono_wide.cuh"

namespace fmm {

namespace {

// packed data of one source cell (level units)
template <typename T>
struct Src {
    T m0, d[3], B2[5], B3[7];
};

template <typename T>
__device__ __forceinline__ void load4(const T *p, T v[4])
{
    if constexpr (kF32<T>) {
        const float4 f = __ldg(reinterpret_cast<const float4 *>(p));
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else if constexpr (kDF<T>) {
        const float4 a = __ldg(reinterpret_cast<const float4 *>(p));
        const float4 b = __ldg(reinterpret_cast<const float4 *>(p) + 1);
        v[0] = dfloat(a.x, a.y); v[1] = dfloat(a.z, a.w);
        v[2] = dfloat(b.x, b.y); v[3] = dfloat(b.z, b.w);
    } else {
        const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
        const double2 b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
        v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
    }
}

__device__ __forceinline__ void unpack_source(const float (&v)[16], Src<float> &s)
{
    s.d[0] = v[0]; s.d[1] = v[1]; s.d[2] = v[2];
    s.m0 = v[3];
#pragma unroll
    for (int k = 0; k < 5; ++k) s.B2[k] = v[4 + k];
#pragma unroll
    for (int q = 0; q < 7; ++q) s.B3[q] = v[9 + q];
}

__device__ __forceinline__ void load_source_at(const float *base, Src<float> &s)
{
    float v[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) load4<float>(base + size_t(g) * NCELL * 4, v + 4 * g);
    unpack_source(v, s);
}

// the same for the wide types; base also names the zero row of leaf sources
template <typename T>
__device__ __forceinline__ void load_wide(const T *base, WideSrc<T> &s)
{
    T v[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) load4<T>(base + size_t(g) * NCELL * 4, v + 4 * g);
    s.d[0] = v[0]; s.d[1] = v[1]; s.d[2] = v[2];
    s.m0 = v[3];
#pragma unroll
    for (int k = 0; k < 5; ++k) s.t2[k] = v[4 + k];
#pragma unroll
    for (int q = 0; q < 7; ++q) s.t3[q] = v[9 + q];
}

__device__ __forceinline__ void load_source(const KParams &P, int row, int pi, Src<float> &s)
{
    load_source_at(static_cast<const float *>(P.mp) + (size_t(row) * 4 * NCELL + pi) * 4, s);
}

__device__ __forceinline__ void zero_moments(Src<float> &s)
{
    s.d[0] = s.d[1] = s.d[2] = 0.f;
#pragma unroll
    for (int k = 0; k < 5; ++k) s.B2[k] = 0.f;
#pragma unroll
    for (int q = 0; q < 7; ++q) s.B3[q] = 0.f;
}

// One source (multipole if SRC_MP, else a point mass m0 = s.m0) into a
// multipole target's 16 traceless accumulators and the correction sum
//   S_i += sum_q (B3_B - M0_B a3_A)_q D4[i, q],  a3_A = B3_A / M0_A,
// with the sign of L folded in:
//   L0 -= M0 D0 + B2.D2 - B3.D3,  L1_i -= M0 D1_i + B2.D3[i,.],
//   L2 -= M0 D2,  L3 -= M0 D3.
// Every product goes straight into its chunk sum as one fused multiply-add.
//
// Expansion order 2 (ORDER = 2; truncation n + m <= 2): L0 -= M0 D0 + B2.D2,
// L1 -= M0 D1, L2 -= M0 D2, no L3, and the correction is the dropped
// n = 1, m = 2 term with the target's share added (D3 is odd):
//   S_i -= sum_k (B2_B + M0_B a2_A)_k D3[i, k],  a2_A = B2_A / M0_A
// (aA holds a2_A in its first five entries then).
// WHAT: 1 only the Taylor coefficients, 2 only the correction, 3 both.
template <bool SRC_MP, int ORDER = 3, int WHAT = 3, class LA, class SA>
__device__ __forceinline__ void acc_mp(float Rx, float Ry, float Rz, const Src<float> &s,
                                       const float aA[7], LA &L, SA &S)
{
    DTraceless D;
    D.eval<ORDER == 3>(Rx, Ry, Rz);
    const float nm0 = -s.m0;
    if constexpr (WHAT & 1) {
        float a = fmaf(nm0, D.D0, L.part[0]);
        if (SRC_MP) {
#pragma unroll
            for (int k = 0; k < 5; ++k) a = fmaf(-s.B2[k], D.D2[k], a);
            if (ORDER == 3) {
#pragma unroll
                for (int q = 0; q < 7; ++q) a = fmaf(s.B3[q], D.D3[q], a);
            }
        }
        L.part[0] = a;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            float b = fmaf(nm0, D.D1[i], L.part[1 + i]);
            if (SRC_MP && ORDER == 3) {
#pragma unroll
                for (int k = 0; k < 5; ++k) b = fmaf(-s.B2[k], D.d3slice(i, k), b);
            }
            L.part[1 + i] = b;
        }
    }
    if constexpr (ORDER == 2) {
        if constexpr (WHAT & 1)
#pragma unroll
            for (int k = 0; k < 5; ++k) L.part[4 + k] = fmaf(nm0, D.D2[k], L.part[4 + k]);
        if constexpr (WHAT & 2) {
            float wn[5];
#pragma unroll
            for (int k = 0; k < 5; ++k) wn[k] = SRC_MP ? fmaf(nm0, aA[k], -s.B2[k]) : nm0 * aA[k];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                float c = S.part[i];
#pragma unroll
                for (int k = 0; k < 5; ++k) c = fmaf(wn[k], D.d3slice(i, k), c);
                S.part[i] = c;
            }
        }
    } else {
        if constexpr (WHAT & 1) {
            // orders 2-3 (12 components): the pairs in which the derivative
            // tensors come out of DTraceless (xx yy | xz yz of D2, xxx yyy
            // | xxz yyz of D3) on the paired FP32 pipe (fma.rn.f32x2: each half
            // rounds as fmaf does), the other four scalar
            constexpr int pair_a[4] = {4, 7, 9, 11}, pair_b[4] = {5, 8, 14, 15};
            const float dv[16] = {0.f, 0.f, 0.f, 0.f, D.D2[0], D.D2[1], D.D2[2], D.D2[3],
                                  D.D2[4], D.D3[0], D.D3[1], D.D3[2], D.D3[3], D.D3[4],
                                  D.D3[5], D.D3[6]};
            const float2 nm2 = make_float2(nm0, nm0);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int a = pair_a[j], b = pair_b[j];
                const float2 r = __ffma2_rn(nm2, make_float2(dv[a], dv[b]),
                                            make_float2(L.part[a], L.part[b]));
                L.part[a] = r.x;
                L.part[b] = r.y;
            }
            L.part[6] = fmaf(nm0, dv[6], L.part[6]);
            L.part[10] = fmaf(nm0, dv[10], L.part[10]);
            L.part[12] = fmaf(nm0, dv[12], L.part[12]);
            L.part[13] = fmaf(nm0, dv[13], L.part[13]);
        }
        if constexpr (WHAT & 2) {
            float w[7];
#pragma unroll
            for (int q = 0; q < 7; ++q) w[q] = SRC_MP ? fmaf(nm0, aA[q], s.B3[q]) : nm0 * aA[q];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                float c = S.part[i];
#pragma unroll
                for (int q = 0; q < 7; ++q) c = fmaf(w[q], D.U[i][q], c);
                S.part[i] = c;
            }
        }
    }
}

// One multipole source into a leaf target (orders 0-1 and the correction;
// the target has no third moment)
// (ORDER = 2: L0 -= M0 D0 + B2.D2, L1 -= M0 D1, S_i -= B2 . D3[i, .])
template <int ORDER = 3>
__device__ __forceinline__ void acc_mx(float Rx, float Ry, float Rz, const Src<float> &s,
                                       Acc<4> &L, Acc<3> &S)
{
    DTraceless D{};
    D.eval<ORDER == 3>(Rx, Ry, Rz);
    float a = -s.m0 * D.D0;
#pragma unroll
    for (int k = 0; k < 5; ++k) a = fmaf(-s.B2[k], D.D2[k], a);
    if (ORDER == 3) {
#pragma unroll
        for (int q = 0; q < 7; ++q) a = fmaf(s.B3[q], D.D3[q], a);
    }
    L.part[0] = L.part[0] + a;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        float b = -s.m0 * D.D1[i];
        float c = S.part[i];
        if constexpr (ORDER == 3) {
#pragma unroll
            for (int k = 0; k < 5; ++k) b = fmaf(-s.B2[k], D.d3slice(i, k), b);
#pragma unroll
            for (int q = 0; q < 7; ++q) c = fmaf(s.B3[q], D.U[i][q], c);
        } else {
#pragma unroll
            for (int k = 0; k < 5; ++k) c = fmaf(-s.B2[k], D.d3slice(i, k), c);
        }
        L.part[1 + i] = L.part[1 + i] + b;
        S.part[i] = c;
    }
}

// target-to-source separation in cell widths, R = (dA - d) - E, in that
// order; x and y go as one pair (the offsets' x and y sit in
// aligned register pairs: first in their 16-byte groups)
__device__ __forceinline__ void separation(const float dA[3], const float d[3], const float4 &E,
                                           float R[3])
{
    const float2 u = fsub2_rn(make_float2(dA[0], dA[1]), make_float2(d[0], d[1]));
    const float2 r = fsub2_rn(u, make_float2(E.x, E.y));
    R[0] = r.x;
    R[1] = r.y;
    R[2] = dA[2] - d[2] - E.z;
}

// own packed data of a multipole target: centre-of-mass offset and
// a3 = B3/M0 (order 3) or a2 = B2/M0 in the first five entries (order 2)
template <int ORDER = 3>
__device__ __forceinline__ void load_target(const KParams &P, int row, int pi, float dA[3], float aA[7])
{
    Src<float> own;
    load_source(P, row, pi, own);
    const float im0 = 1.f / own.m0;
#pragma unroll
    for (int a = 0; a < 3; ++a) dA[a] = own.d[a];
    if (ORDER == 3) {
#pragma unroll
        for (int q = 0; q < 7; ++q) aA[q] = own.B3[q] * im0;
    } else {
#pragma unroll
        for (int q = 0; q < 5; ++q) aA[q] = own.B2[q] * im0;
        aA[5] = aA[6] = 0.f;
    }
}

__device__ __forceinline__ double to_double(float v) { return double(v); }
__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(dfloat v) { return v.to_double(); }

template <class SA>
__device__ __forceinline__ double acc_value(const SA &S, int i)
{
    return to_double(acc_hi(S, i)) + to_double(acc_lo(S, i));
}

// ------------------------------------------------- monopole<-multipole
// One leaf target cell with refined sources (one lane): its own list of
// (packed-moment offset, stencil entry) pairs, orders 0-1 and the correction
// added to what the monopole kernel stored for the cell.
template <typename T, int ORDER = 3>
__device__ __forceinline__ void mx_target(const KParams &P, int t)
{
    const T *mp = static_cast<const T *>(P.mp);
    const int4 tg = __ldg(P.mx_targets + t);       // node, cell, pair offset, count
    const int x = tg.y & 7, y = (tg.y >> 3) & 7, z = tg.y >> 6;
    const int p = (x & 1) + 2 * (y & 1) + 4 * (z & 1);
    const float4 *ent = P.stencil_f + p * P.ent_stride;   // float offsets: no conversions
    using Low = std::conditional_t<kF32<T>, Acc<4>, WideChunked<T, WideLow<T, ORDER>>>;
    Low L;
    Acc<3> S;                               // float only
    L.zero();
    S.zero();
    int done = 0;
    // this lane's pairs, interleaved with its warp's: pair k at base + 32 k + lane;
    // the next pair is fetched while the current one is evaluated
    const int2 *pairs = P.mx_pairs + size_t(tg.z) + (t & 31);
    int2 next = tg.w > 0 ? __ldg(pairs) : make_int2(0, 0);
    for (int k = 0; k < tg.w; ++k) {
        const int2 pr = next;
        if (k + 1 < tg.w) next = __ldg(pairs + size_t(k + 1) * 32);
        const float4 E = __ldg(ent + pr.y);
        if constexpr (kF32<T>) {
            Src<float> src;
            load_source_at(mp + pr.x, src);
            acc_mx<ORDER>(-E.x - src.d[0], -E.y - src.d[1], -E.z - src.d[2], src, L, S);
        } else {
            WideSrc<T> src;
            load_wide<T>(mp + pr.x, src);
            wide_add_leaf<T, ORDER>(wide_sep(T(0), src.d[0], E.x), wide_sep(T(0), src.d[1], E.y),
                                    wide_sep(T(0), src.d[2], E.z), src, L.part);
        }
        if (++done == kChunk) {
            L.flush();
            S.flush();
            done = 0;
        }
    }
    L.flush();
    S.flush();
    const int node = tg.x, cell = tg.y;
    if constexpr (kF32<T>) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const size_t idx = (size_t(node) * NCOMP + k) * NCELL + cell;
            float *Lh = static_cast<float *>(P.L);
            float s, e;
            two_sum(Lh[idx], L.hi[k], s, e);
            const float lo = P.Lc[idx] + L.lo[k] + e;
            const float s2 = s + lo;
            Lh[idx] = s2;
            P.Lc[idx] = lo - (s2 - s);
        }
#pragma unroll
        for (int i = 0; i < 3; ++i)
            P.dL1[(size_t(node) * 3 + i) * NCELL + cell] = acc_value(S, i);
    } else {
        const WideLow<T, ORDER> &A = L.total();
        const T v[4] = {-A.a0, A.a1[0], A.a1[1], A.a1[2]};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const size_t idx = (size_t(node) * NCOMP + k) * NCELL + cell;
            if constexpr (kDF<T>) {
                float *Lh = static_cast<float *>(P.L);
                const dfloat w = dfloat(Lh[idx], P.Lc[idx]) + v[k];
                Lh[idx] = w.hi;
                P.Lc[idx] = w.lo;
            } else {
                static_cast<double *>(P.L)[idx] += v[k];
            }
        }
        T c[3];
        A.correction(c);
#pragma unroll
        for (int i = 0; i < 3; ++i) P.dL1[(size_t(node) * 3 + i) * NCELL + cell] = to_double(c[i]);
    }
}

// ------------------------------------------------------------ mp_kernel
// The far loop of a warp's 32 targets, software-pipelined by hand: while one
// entry is evaluated, the moments of the next are loaded, the window value of
// the one after (which says where its moments are) and the window offset of
// the one after that, so a warp waits for none of the three dependent loads;
// leaf lanes load the zero row.
template <int ORDER, int THREADS>
__device__ __forceinline__ void mp_far_ahead(const KParams &P, const float *W, const float *mp,
                                             const float4 *ent, int base, const float dA[3],
                                             const float a3A[7], SmemAcc<16, 4, THREADS> &L,
                                             SmemAcc<3, 3, THREADS> &S)
{
    const int last = P.n_far - 1;
    float4 E = __ldg(ent);
    float wv = W[base + __float_as_int(E.w)];
    float wv1 = W[base + __float_as_int(__ldg(&ent[min(1, last)].w))];
    int off2 = __float_as_int(__ldg(&ent[min(2, last)].w));
    Src<float> src;
    int idx;
    bool is_mp = window_moments<float>(wv, P.mp_limit, idx);
    load_source_at(mp + (is_mp ? idx : P.mp_limit), src);
    for (int e0 = 0; e0 < P.n_far; e0 += kChunk) {
        const int e1 = min(e0 + kChunk, P.n_far);
        for (int e = e0; e < e1; ++e) {
            Src<float> src1;
            const bool is_mp1 = window_moments<float>(wv1, P.mp_limit, idx);
            load_source_at(mp + (is_mp1 ? idx : P.mp_limit), src1);
            const float wv2 = W[base + off2];
            off2 = __float_as_int(__ldg(&ent[min(e + 3, last)].w));
            const float4 E1 = __ldg(ent + min(e + 1, last));
            if (__any_sync(0xffffffffu, is_mp)) {
                if (!is_mp) src.m0 = wv;
                float R[3];
                separation(dA, src.d, E, R);
                acc_mp<true, ORDER>(R[0], R[1], R[2], src, a3A, L, S);
            } else if (__any_sync(0xffffffffu, window_nonzero<float>(wv))) {
                src.m0 = wv;
                acc_mp<false, ORDER>(dA[0] - E.x, dA[1] - E.y, dA[2] - E.z, src, a3A, L, S);
            }
            src = src1;
            is_mp = is_mp1;
            wv = wv1;
            wv1 = wv2;
            E = E1;
        }
        L.flush();
        S.flush();
    }
}

// The far loop where so few warps share an SM that neither the moment loads nor
// the arithmetic's latency is hidden by other warps: the moments of the next
// DEPTH - 2 entries are in flight to a ring in shared memory (cp.async, zeros for
// leaf lanes; each lane copies and reads its own 64 bytes per entry, so no
// barrier is needed), and two entries are evaluated side by side, their terms
// added in order (an absent source's terms are exact zeros).
// ring: DEPTH entries of four 16-byte groups, 32 lanes apart, from this lane's
template <int ORDER, int WHAT, int DEPTH, int THREADS>
__device__ __forceinline__ void mp_far_staged(const KParams &P, const float *W, const float *mp,
                                              const float4 *ent, int base, const float dA[3],
                                              const float a3A[7], float4 *ring,
                                              SmemAcc<16, 4, THREADS> &L, SmemAcc<3, 3, THREADS> &S)
{
    static_assert(DEPTH % 2 == 0 && DEPTH >= 4 && kChunk % 2 == 0, "pairs");
    const int last = P.n_far - 1;
    // window value of entry i (0, an absent source, past the last)
    auto value = [&](int i, float w) { return i <= last ? W[base + __float_as_int(w)] : 0.f; };
    auto issue = [&](int i, float w) {
        int idx;
        const bool is_mp = window_moments<float>(value(i, w), P.mp_limit, idx);
        const float *src = mp + (is_mp ? idx : P.mp_limit);
        float4 *slot = ring + (i % DEPTH) * 128;
#pragma unroll
        for (int g = 0; g < 4; ++g) cp_async16(slot + 32 * g, src + size_t(g) * NCELL * 4, is_mp);
    };
    for (int i = 0; i < DEPTH - 2; i += 2) {
        issue(i, __ldg(&ent[min(i, last)].w));
        issue(i + 1, __ldg(&ent[min(i + 1, last)].w));
        cp_async_commit();
    }
    float4 E[2] = {__ldg(ent), __ldg(ent + min(1, last))};
    float off[2] = {__ldg(&ent[min(DEPTH - 2, last)].w), __ldg(&ent[min(DEPTH - 1, last)].w)};
    for (int e0 = 0; e0 < P.n_far; e0 += kChunk) {
        const int e1 = min(e0 + kChunk, P.n_far);
        for (int e = e0; e < e1; e += 2) {
            cp_async_wait<DEPTH / 2 - 2>();
            Src<float> src[2];
            float R[2][3];
            bool some = false;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const float wv = value(e + k, E[k].w);
                int idx;
                const bool is_mp = window_moments<float>(wv, P.mp_limit, idx);
                const float4 *slot = ring + ((e + k) % DEPTH) * 128;
                float v[16];
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    const float4 q = slot[32 * g];
                    v[4 * g] = q.x; v[4 * g + 1] = q.y; v[4 * g + 2] = q.z; v[4 * g + 3] = q.w;
                }
                unpack_source(v, src[k]);
                if (!is_mp) src[k].m0 = wv;
                some = some || is_mp || window_nonzero<float>(wv);
                separation(dA, src[k].d, E[k], R[k]);
            }
            // (into the slots of the pair before, whose values have been used)
            issue(e + DEPTH - 2, off[0]);
            issue(e + DEPTH - 1, off[1]);
            cp_async_commit();
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                off[k] = __ldg(&ent[min(e + DEPTH + k, last)].w);
                E[k] = __ldg(ent + min(e + 2 + k, last));
            }
            if (!__any_sync(0xffffffffu, some)) continue;
#pragma unroll
            for (int k = 0; k < 2; ++k)
                acc_mp<true, ORDER, WHAT>(R[k][0], R[k][1], R[k][2], src[k], a3A, L, S);
        }
        if (WHAT & 1) L.flush();
        if (WHAT & 2) S.flush();
    }
    cp_async_wait_all();
}

// Near sources: leaf cells only (refined ones contribute nothing here: their
// children interact one level down); entries are skipped when none of the
// warp's 32 sources is a leaf with mass (skipping exact zeros changes no sum).
template <int ORDER, int WHAT, int THREADS>
__device__ __forceinline__ void mp_near(const KParams &P, const float *W, const float4 *ent, int base,
                                        const float dA[3], const float a3A[7],
                                        SmemAcc<16, 4, THREADS> &L, SmemAcc<3, 3, THREADS> &S)
{
    for (int e0 = P.n_far; e0 < P.n_far + P.n_near; e0 += kChunk) {
        const int e1 = min(e0 + kChunk, P.n_far + P.n_near);
        for (int e = e0; e < e1; ++e) {
            const float4 E = __ldg(ent + e);
            const float wv = W[base + __float_as_int(E.w)];
            Src<float> src;
            src.m0 = window_refined<float>(wv) ? 0.f : wv;
            if (!__any_sync(0xffffffffu, window_nonzero<float>(src.m0))) continue;
            acc_mp<false, ORDER, WHAT>(dA[0] - E.x, dA[1] - E.y, dA[2] - E.z, src, a3A, L, S);
        }
        if (WHAT & 1) L.flush();
        if (WHAT & 2) S.flush();
    }
}

// fmm_step also hands the multipole launch the monopole<-multipole targets:
// once the multipole queue is empty, each warp pulls 32 of them at a time
// from their own queue, which fills the tail that the coarse multipole
// items leave (the monopole kernel, whose results they add to, has
// finished before this launch)
template <int ORDER>
__device__ __forceinline__ void mx_tail(const KParams &P)
{
    const int lane = threadIdx.x & 31;
    while (P.n_mx > 0) {
        int w = 0;
        if (lane == 0) w = atomicAdd(P.mx_counter, 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w * 32 >= P.n_mx) break;
        if (w * 32 + lane < P.n_mx) mx_target<float, ORDER>(P, w * 32 + lane);
    }
}

// PARTS 1: an item is a sub-grid, a warp each parity, both halves (z < 4, z >=
// 4); 2: one half of a sub-grid; 4, WARPS 4: one half of four parities.
// Three CTAs of eight warps per SM (at most 85 registers): the compensation
// pairs, touched once per chunk, live in shared memory after the window.
// AHEAD (mp_far_ahead) takes 112 registers and two such CTAs per SM, WARPS 4
// mp_far_staged: worth it only where the items do not fill the SMs anyway.
constexpr int kMpDepth = 4;      // entries of the ring of WARPS 4
template <int ORDER, int PARTS, bool AHEAD, int WARPS = 8>
__global__ void __launch_bounds__(32 * WARPS, AHEAD || WARPS == 4 ? 2 : 3) mp_kernel(KParams P)
{
    static_assert(WARPS == 8 ? PARTS <= 2 : WARPS == 4 && PARTS == 4, "items per sub-grid");
    constexpr int threads = 32 * WARPS;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *W = reinterpret_cast<float *>(smem_raw);
    float *Cs = W + 8 * P.sub_stride + threadIdx.x;
    __shared__ int s_nbr[27], s_leaf[27], s_row[27], s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cx = lane & 3, cy = (lane >> 2) & 3, cz0 = lane >> 4;
    const float *mass = static_cast<const float *>(P.mass);
    const float *mp = static_cast<const float *>(P.mp);
    for (;;) {
        const int item = pull_item(P.counter, &s_item);
        if (item >= P.n_items) break;
        const int node = P.list[item / PARTS];
        const int p = WARPS == 8 ? warp : 4 * ((item >> 1) & 1) + warp;
        const int px = p & 1, py = (p >> 1) & 1, pz = p >> 2;
        const float4 *ent = P.stencil_f + p * P.ent_stride;   // float offsets: no conversions
        const NodeInfo ti = P.info[node];
        // near sources contribute only if some neighbour is a leaf
        const int any_leaf = __syncthreads_or(load_slots(node, P, s_nbr, s_leaf, s_row));
        stage_window_async<float>(W, s_nbr, s_leaf, mass, P, s_row);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        const int half0 = PARTS == 1 ? 0 : item & 1;
        const int half1 = PARTS == 1 ? 2 : half0 + 1;
        for (int half = half0; half < half1; ++half) {
            const int cz = cz0 + 2 * half;
            const int ax = 2 * cx + px, ay = 2 * cy + py, az = 2 * cz + pz;
            const int base = cx + P.py * cy + P.pz * cz;
            float dA[3], a3A[7];
            load_target<ORDER>(P, ti.mp_row, parity_index(ax, ay, az), dA, a3A);
            SmemAcc<16, 4, threads> L;
            SmemAcc<3, 3, threads> S;
            L.col = Cs;
            S.col = Cs + 4 * 2 * threads;
            L.zero();
            S.zero();
            // Well-separated sources: refined (full moments) or leaf (mass).
            // A vote classifies the warp's 32 sources of one
            // entry: all refined take the moments without a branch, all
            // leaves the mass-only form (the same operations less the zero
            // moments' terms, so the same values), a mix the general form
            // with zero moments for the leaves, and an entry with only
            // absent sources (mass 0) is skipped.
            if constexpr (WARPS == 4) {
                float4 *ring = reinterpret_cast<float4 *>(W + 8 * P.sub_stride + 2 * kMpPairs * threads) +
                               warp * kMpDepth * 128 + lane;
                mp_far_staged<ORDER, 3, kMpDepth>(P, W, mp, ent, base, dA, a3A, ring, L, S);
            } else if constexpr (AHEAD) {
                mp_far_ahead<ORDER>(P, W, mp, ent, base, dA, a3A, L, S);
            } else {
                for (int e0 = 0; e0 < P.n_far; e0 += kChunk) {
                    const int e1 = min(e0 + kChunk, P.n_far);
                    for (int e = e0; e < e1; ++e) {
                        const float4 E = __ldg(ent + e);
                        const float wv = W[base + __float_as_int(E.w)];
                        int idx;
                        const bool is_mp = window_moments<float>(wv, P.mp_limit, idx);
                        const bool all_mp = __all_sync(0xffffffffu, is_mp);
                        Src<float> src;
                        float R[3];
                        if (all_mp) {
                            load_source_at(mp + idx, src);
                            separation(dA, src.d, E, R);
                            acc_mp<true, ORDER>(R[0], R[1], R[2], src, a3A, L, S);
                        } else if (!__any_sync(0xffffffffu, is_mp)) {
                            if (__any_sync(0xffffffffu, window_nonzero<float>(wv))) {
                                src.m0 = wv;
                                acc_mp<false, ORDER>(dA[0] - E.x, dA[1] - E.y,
                                                        dA[2] - E.z, src, a3A, L, S);
                            }
                        } else {
                            if (is_mp) {
                                load_source_at(mp + idx, src);
                            } else {
                                src.m0 = wv;
                                zero_moments(src);
                            }
                            separation(dA, src.d, E, R);
                            acc_mp<true, ORDER>(R[0], R[1], R[2], src, a3A, L, S);
                        }
                    }
                    L.flush();
                    S.flush();
                }
            }
            // skipped when no neighbour is a leaf
            if (any_leaf) mp_near<ORDER, 3>(P, W, ent, base, dA, a3A, L, S);
            const int cell = ax + 8 * ay + 64 * az;
            store_target(P, node, cell, L);
#pragma unroll
            for (int i = 0; i < 3; ++i)
                __stcs(P.dL1 + (size_t(node) * 3 + i) * NCELL + cell, acc_value(S, i));
        }
        __syncthreads();
    }
    mx_tail<ORDER>(P);
}

// Trees with few refined sub-grids, whose time is that of one warp's walk
// through the stencil: two warps share 32 targets (one parity of one half of a
// sub-grid), one forming their Taylor coefficients and one their correction,
// which have no operation in common but the separation's powers.  The walk goes
// from 158 instructions per entry to 100: eight sub-grids below the root (a
// three-level tree's step) 149 -> 137 us, against one warp for both, and
// 137 -> 115 us with mp_far_staged.  Same sums in the same order.
// A CTA is one such pair, an item a sixteenth of a sub-grid.
constexpr int kSplitParts = 16, kSplitThreads = 64, kSplitDepth = 8;
template <int ORDER>
__global__ void __launch_bounds__(kSplitThreads, 2) mp_split_kernel(KParams P)
{
    constexpr int threads = kSplitThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *W = reinterpret_cast<float *>(smem_raw);
    float *Cs = W + 8 * P.sub_stride + threadIdx.x;
    __shared__ int s_nbr[27], s_leaf[27], s_row[27], s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    float4 *ring = reinterpret_cast<float4 *>(W + 8 * P.sub_stride + 2 * kMpPairs * threads) +
                   warp * kSplitDepth * 128 + lane;
    const int cx = lane & 3, cy = (lane >> 2) & 3;
    const float *mass = static_cast<const float *>(P.mass);
    const float *mp = static_cast<const float *>(P.mp);
    for (;;) {
        const int item = pull_item(P.counter, &s_item);
        if (item >= P.n_items) break;
        const int node = P.list[item / kSplitParts];
        const int p = (item >> 1) & 7;
        const float4 *ent = P.stencil_f + p * P.ent_stride;
        const NodeInfo ti = P.info[node];
        const int any_leaf = __syncthreads_or(load_slots(node, P, s_nbr, s_leaf, s_row));
        stage_window_async<float>(W, s_nbr, s_leaf, mass, P, s_row);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        const int cz = (lane >> 4) + 2 * (item & 1);
        const int ax = 2 * cx + (p & 1), ay = 2 * cy + ((p >> 1) & 1), az = 2 * cz + (p >> 2);
        const int base = cx + P.py * cy + P.pz * cz, cell = ax + 8 * ay + 64 * az;
        float dA[3], a3A[7];
        load_target<ORDER>(P, ti.mp_row, parity_index(ax, ay, az), dA, a3A);
        SmemAcc<16, 4, threads> L;
        SmemAcc<3, 3, threads> S;
        L.col = Cs;
        S.col = Cs + 4 * 2 * threads;
        L.zero();
        S.zero();
        if (warp == 0) {
            mp_far_staged<ORDER, 1, kSplitDepth>(P, W, mp, ent, base, dA, a3A, ring, L, S);
            if (any_leaf) mp_near<ORDER, 1>(P, W, ent, base, dA, a3A, L, S);
            store_target(P, node, cell, L);
        } else {
            mp_far_staged<ORDER, 2, kSplitDepth>(P, W, mp, ent, base, dA, a3A, ring, L, S);
            if (any_leaf) mp_near<ORDER, 2>(P, W, ent, base, dA, a3A, L, S);
#pragma unroll
            for (int i = 0; i < 3; ++i)
                __stcs(P.dL1 + (size_t(node) * 3 + i) * NCELL + cell, acc_value(S, i));
        }
        __syncthreads();
    }
    mx_tail<ORDER>(P);
}

// ---------------------------------------------------------- mpw_kernel
// The multipole kernel of the wide types (double, double-float; the
// interaction and its sums are in fmm_wide.cuh).  Bound by the FP64 pipe
// (double) or the FP32 pipe (double-float): one CTA per SM is enough, and
// registers go to the 34 sums.  One loop takes far and near entries alike
// (near ones count leaf sources only), so the large body is compiled once;
// its second half, the moments, is skipped for entries without a refined
// source in the warp, and entries with absent sources only altogether.
// CTAs of four warps: three per SM in double-float (at most 168 registers),
// whose dependent chains leave the pipe idle with two warps a scheduler; two
// in double, which fills its pipe with those and needs the registers for the
// chunk sums.
//   PARTS 2, 4: an item is four of a sub-grid's eight parities (one z parity),
//     a warp each, in both halves (z < 4, z >= 4) or one of them;
//   PARTS 16: an item is one half of one parity, 32 cells, whose stencil
//     entries the four warps share out (every fourth entry), the sums added
//     through shared memory in a fixed order: for trees with too few refined
//     nodes to fill the SMs otherwise.
constexpr int kWideThreads = 128;
template <typename T>
__device__ __forceinline__ T wide_shfl_xor(T v, int mask)
{
    if constexpr (kDF<T>)
        return dfloat(__shfl_xor_sync(0xffffffffu, v.hi, mask), __shfl_xor_sync(0xffffffffu, v.lo, mask));
    else
        return __shfl_xor_sync(0xffffffffu, v, mask);
}
// the sums of WideAcc as an array
template <int ORDER>
constexpr int kWideSums = ORDER == 3 ? 34 : 22;

template <typename T, int ORDER>
__device__ __forceinline__ void store_wide(const KParams &P, int node, int cell, const T L[16], const T S[3])
{
    T zero[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) zero[k] = T(0);
    store_target_values<T>(P, node, cell, L, zero);
#pragma unroll
    for (int i = 0; i < 3; ++i)
        __stcs(P.dL1 + (size_t(node) * 3 + i) * NCELL + cell, to_double(S[i]));
}

template <typename T, int ORDER, int PARTS>
__global__ void __launch_bounds__(kWideThreads, kDF<T> ? 3 : 2) mpw_kernel(KParams P)
{
    static_assert(PARTS == 2 || PARTS == 4 || PARTS == 16, "items per sub-grid");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    T *W = reinterpret_cast<T *>(smem_raw);
    __shared__ int s_nbr[27], s_leaf[27], s_row[27], s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cx = lane & 3, cy = (lane >> 2) & 3, cz0 = lane >> 4;
    const T *mass = static_cast<const T *>(P.mass);
    const T *mp = static_cast<const T *>(P.mp);
    for (;;) {
        const int item = pull_item(P.counter, &s_item);
        if (item >= P.n_items) break;
        const int node = P.list[item / PARTS];
        const NodeInfo ti = P.info[node];
        // near sources contribute only if some neighbour is a leaf
        const int any_leaf = __syncthreads_or(load_slots(node, P, s_nbr, s_leaf, s_row));
        stage_window_async<T>(W, s_nbr, s_leaf, mass, P, s_row);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        const int p = PARTS == 16 ? (item >> 1) & 7 : 4 * (item / (PARTS / 2) & 1) + warp;
        const int px = p & 1, py = (p >> 1) & 1, pz = p >> 2;
        const float4 *ent = P.stencil_f + p * P.ent_stride;
        const int n_ent = any_leaf ? P.n_far + P.n_near : P.n_far;
        constexpr int step = PARTS == 16 ? kWideThreads / 32 : 1;
        const int half0 = PARTS == 2 ? 0 : item & 1;
        const int half1 = PARTS == 2 ? 2 : half0 + 1;
        for (int half = half0; half < half1; ++half) {
            const int cz = cz0 + 2 * half;
            const int ax = 2 * cx + px, ay = 2 * cy + py, az = 2 * cz + pz;
            const int base = cx + P.py * cy + P.pz * cz;
            const T *own_at = mp + (size_t(ti.mp_row) * 4 * NCELL + parity_index(ax, ay, az)) * 4;
            T dA[4];
            load4<T>(own_at, dA);
            WideChunked<T, WideAcc<T, ORDER>> C;
            C.zero();
            int done = 0;
            for (int e = PARTS == 16 ? warp : 0; e < n_ent; e += step) {
                const float4 E = __ldg(ent + e);
                T wv = W[base + __float_as_int(E.w)];
                int idx;
                bool is_mp = window_moments<T>(wv, P.mp_limit, idx);
                if (e >= P.n_far) {
                    if (window_refined<T>(wv)) wv = T(0);
                    is_mp = false;
                }
                if (!__any_sync(0xffffffffu, window_nonzero<T>(wv))) continue;
                const bool any_mp = __any_sync(0xffffffffu, is_mp);
                WideSrc<T> src;
                T m = wv;
                if (any_mp) {
                    // leaf lanes read zero moments from the zero row
                    load_wide<T>(mp + (is_mp ? idx : P.mp_limit), src);
                    if (is_mp) m = src.m0;
                } else {
                    src.d[0] = src.d[1] = src.d[2] = T(0);
                }
                C.part.add(wide_sep(dA[0], src.d[0], E.x), wide_sep(dA[1], src.d[1], E.y),
                           wide_sep(dA[2], src.d[2], E.z), m, src, any_mp);
                if (++done == kChunk) {
                    C.flush();
                    done = 0;
                }
            }
            C.flush();
            WideAcc<T, ORDER> &A = C.total();
            if (PARTS == 16) {
                // the upper half of the warps hand their sums to the lower, twice
                constexpr int NS = kWideSums<ORDER>;
                T *sum = reinterpret_cast<T *>(&A);
                for (int w = kWideThreads / 64; w > 0; w >>= 1) {
                    __syncthreads();                // the window, or the last round, is done with
                    if (warp >= w && warp < 2 * w)
#pragma unroll
                        for (int k = 0; k < NS; ++k) W[((warp - w) * NS + k) * 32 + lane] = sum[k];
                    __syncthreads();
                    if (warp < w)
#pragma unroll
                        for (int k = 0; k < NS; ++k) sum[k] += W[(warp * NS + k) * 32 + lane];
                }
            }
            if (PARTS != 16 || warp == 0) {
                WideSrc<T> own;
                load_wide<T>(own_at, own);
                T L[16], S[3];
                A.finish(own, L, S);
                store_wide<T, ORDER>(P, node, ax + 8 * ay + 64 * az, L, S);
            }
        }
        __syncthreads();
    }
    // as in mp_kernel: fmm_step's monopole<-multipole targets fill the tail
    if (P.n_mx > 0) {
        for (;;) {
            int w = 0;
            if (lane == 0) w = atomicAdd(P.mx_counter, 1);
            w = __shfl_sync(0xffffffffu, w, 0);
            if (w * 32 >= P.n_mx) break;
            if (w * 32 + lane < P.n_mx) mx_target<T, ORDER>(P, w * 32 + lane);
        }
    }
}

// ----------------------------------------------------------- mp2_kernel
// The multipole kernel (float) with each thread's two target cells (z and
// z + 4 of one parity) walked through the stencil together instead of one
// after the other: one stencil-entry load serves both, and the two cells'
// independent loads and arithmetic interleave, so each warp has twice the
// work in flight between its dependent steps.  Two CTAs per SM (at most 128
// registers) and both cells' compensation pairs in shared memory.  Every
// cell's operations and their order are those of mp_kernel, so the results
// are the same bits.
constexpr int kMp2Pairs = 2 * kMpPairs;

__device__ __forceinline__ void mp2_source(const KParams &P, const float *mp, float wv, Src<float> &src)
{
    // masses are not negative, so a mass's decoded offset is out of range
    const unsigned idx = unsigned(-1 - __float_as_int(wv));
    if (idx < unsigned(P.mp_limit)) {
        load_source_at(mp + idx, src);
    } else {
        src.m0 = wv;
        zero_moments(src);
    }
}

__global__ void __launch_bounds__(kThreads, 2) mp2_kernel(KParams P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float *W = reinterpret_cast<float *>(smem_raw);
    float *Cs = W + 8 * P.sub_stride + threadIdx.x;
    __shared__ int s_nbr[27], s_leaf[27], s_row[27], s_item;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp;
    const int px = p & 1, py = (p >> 1) & 1, pz = p >> 2;
    const int cx = lane & 3, cy = (lane >> 2) & 3, cz0 = lane >> 4;
    const float4 *ent = P.stencil_f + p * P.ent_stride;
    const float *mass = static_cast<const float *>(P.mass);
    const float *mp = static_cast<const float *>(P.mp);
    for (;;) {
        const int item = pull_item(P.counter, &s_item);
        if (item >= P.n_items) break;
        const int node = P.list[item];
        const NodeInfo ti = P.info[node];
        const int any_leaf = __syncthreads_or(load_slots(node, P, s_nbr, s_leaf, s_row));
        stage_window_async<float>(W, s_nbr, s_leaf, mass, P, s_row);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        const int ax = 2 * cx + px, ay = 2 * cy + py;
        const int az0 = 2 * cz0 + pz, az1 = az0 + 4;
        const int base0 = cx + P.py * cy + P.pz * cz0, base1 = base0 + 2 * P.pz;
        float dA0[3], a3A0[7], dA1[3], a3A1[7];
        load_target<3>(P, ti.mp_row, parity_index(ax, ay, az0), dA0, a3A0);
        load_target<3>(P, ti.mp_row, parity_index(ax, ay, az1), dA1, a3A1);
        SmemAcc<16, 4> L0, L1;
        SmemAcc<3> S0, S1;
        L0.col = Cs;
        S0.col = Cs + 4 * 2 * kThreads;
        L1.col = Cs + kMpPairs * 2 * kThreads;
        S1.col = Cs + (kMpPairs + 4) * 2 * kThreads;
        L0.zero();
        S0.zero();
        L1.zero();
        S1.zero();
        for (int e0 = 0; e0 < P.n_far; e0 += kChunk) {
            const int e1 = min(e0 + kChunk, P.n_far);
            for (int e = e0; e < e1; ++e) {
                const float4 E = __ldg(ent + e);
                const int woff = __float_as_int(E.w);
                const float w0 = W[base0 + woff], w1 = W[base1 + woff];
                const unsigned i0 = unsigned(-1 - __float_as_int(w0));
                const unsigned i1 = unsigned(-1 - __float_as_int(w1));
                Src<float> s0, s1;
                // the warp's 64 sources all refined: the moments without a
                // branch (the same values as the general form)
                if (__all_sync(0xffffffffu, i0 < unsigned(P.mp_limit) && i1 < unsigned(P.mp_limit))) {
                    load_source_at(mp + i0, s0);
                    load_source_at(mp + i1, s1);
                } else {
                    mp2_source(P, mp, w0, s0);
                    mp2_source(P, mp, w1, s1);
                }
                float R0[3], R1[3];
                separation(dA0, s0.d, E, R0);
                separation(dA1, s1.d, E, R1);
                acc_mp<true>(R0[0], R0[1], R0[2], s0, a3A0, L0, S0);
                acc_mp<true>(R1[0], R1[1], R1[2], s1, a3A1, L1, S1);
            }
            L0.flush();
            S0.flush();
            L1.flush();
            S1.flush();
        }
        for (int e0 = P.n_far; any_leaf && e0 < P.n_far + P.n_near; e0 += kChunk) {
            const int e1 = min(e0 + kChunk, P.n_far + P.n_near);
            for (int e = e0; e < e1; ++e) {
                const float4 E = __ldg(ent + e);
                const int woff = __float_as_int(E.w);
                const float w0 = W[base0 + woff], w1 = W[base1 + woff];
                Src<float> s0, s1;
                s0.m0 = unsigned(-1 - __float_as_int(w0)) < unsigned(P.mp_limit) ? 0.f : w0;
                s1.m0 = unsigned(-1 - __float_as_int(w1)) < unsigned(P.mp_limit) ? 0.f : w1;
                if (!__any_sync(0xffffffffu, s0.m0 != 0.f || s1.m0 != 0.f)) continue;
                acc_mp<false>(dA0[0] - E.x, dA0[1] - E.y, dA0[2] - E.z, s0, a3A0, L0, S0);
                acc_mp<false>(dA1[0] - E.x, dA1[1] - E.y, dA1[2] - E.z, s1, a3A1, L1, S1);
            }
            L0.flush();
            S0.flush();
            L1.flush();
            S1.flush();
        }
        const int cell0 = ax + 8 * ay + 64 * az0, cell1 = ax + 8 * ay + 64 * az1;
        store_target(P, node, cell0, L0);
        store_target(P, node, cell1, L1);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            P.dL1[(size_t(node) * 3 + i) * NCELL + cell0] = acc_value(S0, i);
            P.dL1[(size_t(node) * 3 + i) * NCELL + cell1] = acc_value(S1, i);
        }
        __syncthreads();
    }
    mx_tail<3>(P);
}

// ---------------------------------------------------------- mono_kernel
// Leaf target, leaf sources: R = -o exactly, so L0 += c0(o) m and
// L1 += c1(o) m with per-offset weights c0 = -1/|o|, c1 = -o/|o|^3.
// Every parity's stencil is parity 0's reflected along its odd axes, so a
// warp of parity p walks parity 0's entries, reflected (mono_woff holds
// their window offsets), and one weight table (parity 0's) serves all eight
// warps: the warp accumulates with parity 0's first-order weights and flips
// the signs of its L1 components along p's odd axes at the end (exact).  The
// table and the window offsets sit in shared memory, loaded once per CTA;
// every access to them is a warp-uniform broadcast.
// (Mixed precision; the wide types' kernel is in fmm_mono_wide.cuh.)
// Each pass takes NB sub-grids (consecutive in the cost-sorted queue), each
// with its own halo window, staged by cp.async so that every load of the
// window is in flight at once; every thread holds two target cells (z and
// z+4 of one parity) per sub-grid, so each weight feeds 2 NB cells.
// src = the entry's source of this thread's first target cell; the NB windows
// are WSTRIDE apart and the second target cell DZ1 further on (compile-time
// offsets, folded into the shared-memory loads)
template <int NB, int WSTRIDE, int DZ1>
__device__ __forceinline__ void mono_entry(const float *src, const float *coef, int e,
                                           Acc<4> (&A)[NB], Acc<4> (&B)[NB])
{
    const float4 c4 = *reinterpret_cast<const float4 *>(coef + 4 * e);
    const float c[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
    for (int b = 0; b < NB; ++b) {
        const float m0 = src[b * WSTRIDE];
        const float m1 = src[b * WSTRIDE + DZ1];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            A[b].part[k] = fmaf(c[k], m0, A[b].part[k]);
            B[b].part[k] = fmaf(c[k], m1, B[b].part[k]);
        }
    }
}

__device__ __forceinline__ const float *byte_offset(const float *p, unsigned bytes)
{
    return reinterpret_cast<const float *>(reinterpret_cast<const char *>(p) + bytes);
}

// dynamic shared memory of mono_kernel<NB, R>: NB windows, the weight table
// of parity 0 and the window offsets of all parities
inline size_t mono_smem_bytes(int nb, size_t window_bytes, int ent_stride, bool packed)
{
    return nb * window_bytes + size_t(ent_stride) * 4 * sizeof(float) +
           size_t(8) * ent_stride * (packed ? sizeof(uint16_t) : sizeof(int));
}

// PACKED: the window offsets stay 16-bit in shared memory and are read eight
// to a load.  Shared-memory wavefronts bound the loop: five per entry and warp
// instead of six.  The unpacking costs a little latency per chunk, so only
// trees with many passes per CTA use it (launch_mono_r).
template <int NB, int RR, bool PACKED>
__global__ void __launch_bounds__(kThreads) mono_kernel(KParams P)
{
    using G = WinGeo<RR>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int wstride = 8 * G::SUB_STRIDE;
    float *W = reinterpret_cast<float *>(smem_raw);
    float *s_coef = W + NB * wstride;
    using Off = std::conditional_t<PACKED, uint16_t, int>;
    Off *s_woff = reinterpret_cast<Off *>(s_coef + 4 * P.ent_stride);
    __shared__ int s_nbr[NB][27], s_leaf[NB][27], s_row[NB][27], s_item;
    const int n_ent = P.n_far + P.n_near;
    {
        const float *gcoef = P.coef;                              // parity 0's
        for (int i = threadIdx.x; i < 4 * n_ent; i += blockDim.x) s_coef[i] = __ldg(gcoef + i);
        if constexpr (PACKED) {                        // eight offsets each
            for (int i = threadIdx.x; i < P.ent_stride; i += blockDim.x)
                reinterpret_cast<uint4 *>(s_woff)[i] =
                    __ldg(reinterpret_cast<const uint4 *>(P.mono_woff16) + i);
        } else {
            for (int i = threadIdx.x; i < 8 * P.ent_stride; i += blockDim.x)
                s_woff[i] = __ldg(P.mono_woff + i);
        }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = warp;
    const int px = p & 1, py = (p >> 1) & 1, pz = p >> 2;
    const int cx = lane & 3, cy = (lane >> 2) & 3, cz = lane >> 4;
    const Off *woff = s_woff + p * P.ent_stride;
    const float *mass = static_cast<const float *>(P.mass);
    const int base0 = cx + G::PY * cy + G::PZ * cz;
    constexpr int dz1 = 2 * G::PZ;              // the second target cell, z + 4
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(P.counter, NB);
        __syncthreads();
        const int item0 = s_item;
        if (item0 >= P.n_items) break;
        int nodes[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) nodes[b] = item0 + b < P.n_items ? P.list[item0 + b] : -1;
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (nodes[b] >= 0) load_slots(nodes[b], P, s_nbr[b], s_leaf[b], s_row[b]);
        __syncthreads();
#pragma unroll
        for (int b = 0; b < NB; ++b)
            if (nodes[b] >= 0) stage_window_async<float, RR>(W + b * wstride, s_nbr[b], s_leaf[b], mass, P);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        Acc<4> A[NB], B[NB];
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            A[b].zero();
            B[b].zero();
        }
        // 32 entries per compensated chunk (the TwoSum folds are a
        // fifth of this kernel's instructions at 16)
        constexpr int chunk = 2 * kChunk;
        int e = 0;
        for (; e + chunk <= n_ent; e += chunk) {
            if constexpr (PACKED) {
#pragma unroll
                for (int j = 0; j < chunk; j += 8) {
                    const uint4 o = *reinterpret_cast<const uint4 *>(woff + e + j);
                    const unsigned w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const unsigned off = i % 2 ? w[i / 2] >> 16 : w[i / 2] & 0xffffu;
                        mono_entry<NB, wstride, dz1>(byte_offset(W + base0, off), s_coef, e + j + i, A, B);
                    }
                }
            } else {
#pragma unroll
                for (int j = 0; j < chunk; ++j)
                    mono_entry<NB, wstride, dz1>(W + base0 + woff[e + j], s_coef, e + j, A, B);
            }
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                A[b].flush();
                B[b].flush();
            }
        }
        for (; e < n_ent; ++e)
            mono_entry<NB, wstride, dz1>(PACKED ? byte_offset(W + base0, woff[e]) : W + base0 + woff[e],
                                         s_coef, e, A, B);
        const int ax = 2 * cx + px, ay = 2 * cy + py;
        const int cell0 = ax + 8 * ay + 64 * (2 * cz + pz);
        const int cell1 = cell0 + 64 * 4;
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            if (nodes[b] < 0) continue;
            A[b].flush();
            B[b].flush();
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                // first-order weights were parity 0's: undo the reflection
                const bool flip = k > 0 && ((p >> (k - 1)) & 1);
                const float ah = acc_hi(A[b], k), al = acc_lo(A[b], k);
                const float bh = acc_hi(B[b], k), bl = acc_lo(B[b], k);
                store_L<float>(P, nodes[b], k, cell0, flip ? -ah : ah, flip ? -al : al);
                store_L<float>(P, nodes[b], k, cell1, flip ? -bh : bh, flip ? -bl : bl);
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                __stcs(P.dL1 + (size_t(nodes[b]) * 3 + i) * NCELL + cell0, 0.0);
                __stcs(P.dL1 + (size_t(nodes[b]) * 3 + i) * NCELL + cell1, 0.0);
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ mx_kernel
// Leaf targets, refined sources (monopole<-multipole): orders 0-1 and the
// correction (the target has no third moment).  Adds to what mono_kernel
// stored for the same cells, so it runs after it on the same stream.  Few
// targets of a node see refined sources, and those see few (16 on average
// on the workloads), so instead of walking every stencil entry with most
// lanes masked off, each lane takes one target cell and walks that cell's
// own list of (packed-moment offset, stencil entry) pairs, built on the
// host; targets are sorted by list length, so a warp's lanes finish together,
// and a warp's lists are interleaved, so each step of the walk reads the
// warp's 32 pairs as one contiguous block.
template <typename T, int ORDER>
__global__ void __launch_bounds__(kThreads) mx_kernel(KParams P)
{
    const int lane = threadIdx.x & 31;
    const int warps = int(gridDim.x) * (kThreads / 32);
    for (int w = int(blockIdx.x) * (kThreads / 32) + (threadIdx.x >> 5); w * 32 < P.n_items;
         w += warps) {
        const int t = w * 32 + lane;
        if (t < P.n_items) mx_target<T, ORDER>(P, t);
    }
}

// ---------------------------------------------------------- root_kernel
// Level 1 holds one node per tree and every pair is a candidate: a refined
// root evaluates its well-separated pairs, a leaf root all pairs.  The
// 512 x 511 pairs of one root are spread over 16 CTAs of 32 targets, each
// target's 512 sources over 8 warps; the 8 partial sums are folded in a
// fixed order (deterministic).
constexpr int kRootSlices = 8;
constexpr int kRootThreads = 32 * kRootSlices;
constexpr int kRootGroups = NCELL / 32;

template <int ORDER>
__global__ void __launch_bounds__(kRootThreads) root_kernel(KParams P)
{
    constexpr int NV = 16 + 3;                      // L (traceless), S
    __shared__ float sh_hi[kRootSlices][NV][32];
    __shared__ float sh_lo[kRootSlices][NV][32];
    const int node = P.list[blockIdx.x];
    const NodeInfo ti = P.info[node];
    const bool leaf = ti.leaf_row >= 0;
    const float *mass = static_cast<const float *>(P.mass);
    const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
    const int cell = blockIdx.y * 32 + lane;
    const int ax = cell & 7, ay = (cell >> 3) & 7, az = cell >> 6;
    float dA[3] = {0.f, 0.f, 0.f}, a3A[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (!leaf) load_target<ORDER>(P, ti.mp_row, parity_index(ax, ay, az), dA, a3A);
    Acc<16> L;
    Acc<3> S;
    L.zero();
    S.zero();
    int done = 0;
    const int b0 = slice * (NCELL / kRootSlices);
    for (int b = b0; b < b0 + NCELL / kRootSlices; ++b) {
        const int ox = (b & 7) - ax, oy = ((b >> 3) & 7) - ay, oz = (b >> 6) - az;
        const bool far = ox * ox + oy * oy + oz * oz >= P.far_o2;
        if (b == cell || !(far || leaf)) continue;
        const int pi = parity_index(b & 7, (b >> 3) & 7, b >> 6);
        Src<float> src;
        if (!leaf) {
            load_source(P, ti.mp_row, pi, src);
        } else {
            src.m0 = mass[size_t(node) * NCELL + pi];
            zero_moments(src);
        }
        acc_mp<true, ORDER>(dA[0] - src.d[0] - float(ox), dA[1] - src.d[1] - float(oy),
                        dA[2] - src.d[2] - float(oz), src, a3A, L, S);
        if (++done == kChunk) {
            L.flush();
            S.flush();
            done = 0;
        }
    }
    L.flush();
    S.flush();
    for (int k = 0; k < 16; ++k) {
        sh_hi[slice][k][lane] = acc_hi(L, k);
        sh_lo[slice][k][lane] = acc_lo(L, k);
    }
    for (int i = 0; i < 3; ++i) {
        sh_hi[slice][16 + i][lane] = acc_hi(S, i);
        sh_lo[slice][16 + i][lane] = acc_lo(S, i);
    }
    __syncthreads();
    if (slice != 0) return;
    float Fh[NV], Fl[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        float hi = 0.f, lo = 0.f;
        for (int sl = 0; sl < kRootSlices; ++sl) {
            float sum, err;
            two_sum(hi, sh_hi[sl][k][lane], sum, err);
            hi = sum;
            lo += err + sh_lo[sl][k][lane];
        }
        Fh[k] = hi;
        Fl[k] = lo;
    }
    if (leaf) {
        for (int k = 0; k < 4; ++k) store_L<float>(P, node, k, cell, Fh[k], Fl[k]);
    } else {
        store_target_values<float>(P, node, cell, Fh, Fl);
    }
    for (int i = 0; i < 3; ++i)
        P.dL1[(size_t(node) * 3 + i) * NCELL + cell] = to_double(Fh[16 + i]) + to_double(Fl[16 + i]);
}

// The root of the wide types, whose arithmetic fills an SM: four targets per
// CTA and 128 CTAs, so that one root spreads over most SMs (16 CTAs of 32
// targets took 741 us in FP64 and 150 us in double-float).  The 512 sources
// of a target are shared out over 64 threads, eight each; their sums are
// added by shuffles within a warp and in a fixed order across the warps.
constexpr int kRootwTargets = 4;

template <typename T, int ORDER>
__global__ void __launch_bounds__(kThreads) rootw_kernel(KParams P)
{
    constexpr int NS = kWideSums<ORDER>, NW = kThreads / 32;
    static_assert(sizeof(WideAcc<T, ORDER>) == NS * sizeof(T), "sums of WideAcc");
    __shared__ T sh[NW][NS][kRootwTargets];
    const int node = P.list[blockIdx.x];
    const NodeInfo ti = P.info[node];
    const bool leaf = ti.leaf_row >= 0;
    const T *mass = static_cast<const T *>(P.mass);
    const T *mp = static_cast<const T *>(P.mp);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int cell = blockIdx.y * kRootwTargets + (lane & 3);
    const int slice = warp * 8 + (lane >> 2);
    const int ax = cell & 7, ay = (cell >> 3) & 7, az = cell >> 6;
    const T *row = leaf ? mp : mp + size_t(ti.mp_row) * 4 * NCELL * 4;
    const T *own_at = row + parity_index(ax, ay, az) * 4;
    T dA[4] = {T(0), T(0), T(0), T(0)};
    if (!leaf) load4<T>(own_at, dA);
    WideAcc<T, ORDER> A;
    A.zero();
    // source x = slot + k: every slice's eight sources are one x row
    const int by = slice & 7, bz = slice >> 3;
    for (int bx = 0; bx < 8; ++bx) {
        const int ox = bx - ax, oy = by - ay, oz = bz - az;
        const int o2 = ox * ox + oy * oy + oz * oz;
        if (o2 == 0 || !(leaf || o2 >= P.far_o2)) continue;
        const int pi = parity_index(bx, by, bz);
        WideSrc<T> src;
        T m;
        if (!leaf) {
            load_wide<T>(row + pi * 4, src);
            m = src.m0;
        } else {
            m = mass[size_t(node) * NCELL + pi];
            src.d[0] = src.d[1] = src.d[2] = T(0);
        }
        A.add(wide_sep(dA[0], src.d[0], float(ox)), wide_sep(dA[1], src.d[1], float(oy)),
              wide_sep(dA[2], src.d[2], float(oz)), m, src, !leaf);
    }
    A.flush();
    T *sum = reinterpret_cast<T *>(&A);
#pragma unroll
    for (int k = 0; k < NS; ++k) {
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) sum[k] += wide_shfl_xor(sum[k], off);
        if (lane < kRootwTargets) sh[warp][k][lane] = sum[k];
    }
    __syncthreads();
    // (one thread per value and target adds the eight warps' sums)
    for (int i = threadIdx.x; i < NS * kRootwTargets; i += kThreads) {
        const int k = i / kRootwTargets, t = i % kRootwTargets;
        T v = sh[0][k][t];
#pragma unroll
        for (int w = 1; w < NW; ++w) v += sh[w][k][t];
        sh[0][k][t] = v;
    }
    __syncthreads();
    if (threadIdx.x >= kRootwTargets) return;
#pragma unroll
    for (int k = 0; k < NS; ++k) sum[k] = sh[0][k][threadIdx.x];
    if (leaf) {
        store_L<T>(P, node, 0, cell, -A.low.a0, T(0));
        for (int i = 0; i < 3; ++i) store_L<T>(P, node, 1 + i, cell, A.low.a1[i], T(0));
        for (int i = 0; i < 3; ++i) P.dL1[(size_t(node) * 3 + i) * NCELL + cell] = 0.0;
        return;
    }
    WideSrc<T> own;
    load_wide<T>(own_at, own);
    T L[16], S[3];
    A.finish(own, L, S);
    store_wide<T, ORDER>(P, node, cell, L, S);
}

// ---------------------------------------------------------- launching
// opt-in dynamic shared memory of a kernel, raised once to the largest size
// asked for so far
template <typename Kern>
cudaError_t allow_smem(Kern k, size_t bytes, size_t &done)
{
    if (bytes <= done) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e == cudaSuccess) done = bytes;
    return e;
}

template <typename T>
struct Kernels {
    // the wide types' multipole kernel, PARTS items per sub-grid
    template <int ORDER, int PARTS>
    static cudaError_t mpw(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mpw_kernel<T, ORDER, PARTS>, bytes, done);
    }
    template <int ORDER, int PARTS, bool AHEAD, int WARPS>
    static cudaError_t mp(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mp_kernel<ORDER, PARTS, AHEAD, WARPS>, bytes, done);
    }
    template <int ORDER>
    static cudaError_t mp_split(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mp_split_kernel<ORDER>, bytes, done);
    }
    static cudaError_t mp2(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mp2_kernel, bytes, done);
    }
    template <int NB, int RR, bool PACKED>
    static cudaError_t mono(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mono_kernel<NB, RR, PACKED>, bytes, done);
    }
    template <int PLANES>
    static cudaError_t mono_wide(size_t bytes)
    {
        static size_t done = 0;
        return allow_smem(mono_wide_kernel<T, PLANES>, bytes, done);
    }
};

// persistent grid: SMs x resident CTAs (optionally capped by the tuning)
template <typename Kern>
int persistent_grid(Kern k, size_t smem, int64_t items, int sms, int cap_per_sm,
                    int threads = kThreads)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, threads, smem) != cudaSuccess ||
        per_sm < 1)
        per_sm = 1;
    if (cap_per_sm > 0 && cap_per_sm < per_sm) per_sm = cap_per_sm;
    int64_t g = int64_t(per_sm) * sms;
    return int(items < g ? items : g);
}

template <int NB, int RR, bool PACKED>
cudaError_t launch_mono_p(const KParams &K, size_t wbytes, int sms, int cap, cudaStream_t s)
{
    const size_t bytes = mono_smem_bytes(NB, wbytes, K.ent_stride, PACKED);
    cudaError_t e = Kernels<float>::mono<NB, RR, PACKED>(bytes);
    if (e != cudaSuccess) return e;
    const int64_t passes = (K.n_items + NB - 1) / NB;
    int g = persistent_grid(mono_kernel<NB, RR, PACKED>, bytes, passes, sms, cap);
    if (PACKED) g = std::min(g, 5 * sms / 2);
    mono_kernel<NB, RR, PACKED><<<g, kThreads, bytes, s>>>(K);
    return cudaGetLastError();
}

// Packed offsets for pairs of sub-grids and at least eight passes an SM: with
// 15 passes (4572 leaf sub-grids) the same-level pass takes 818 -> 801 us and
// a theta = 0.35 step 2238 -> 2177 us, with five (1457) a step 399 -> 408 us.
// The smaller table lets a third CTA onto an SM at theta = 0.5, but only half
// of the SMs get one (level-7 tree's step 2439 -> 2413 us): beside three CTAs
// on each SM the upward pass finds no room (2461 us).
template <int NB, int RR>
cudaError_t launch_mono_r(const KParams &K, size_t wbytes, int sms, int cap, cudaStream_t s)
{
    // the compile-time window geometry must be the host's
    using G = WinGeo<RR>;
    if (K.reach != G::R || K.py != G::PY || K.pz != G::PZ || K.sub_stride != G::SUB_STRIDE)
        return cudaErrorInvalidValue;
    if constexpr (NB == 2)
        if (K.n_items >= 8 * int64_t(sms) * NB) return launch_mono_p<NB, RR, true>(K, wbytes, sms, cap, s);
    return launch_mono_p<NB, RR, false>(K, wbytes, sms, cap, s);
}

// theta in (0.25, 1/sqrt(3)] gives reach 2 floor(1/theta) + 1 = 3, 5 or 7
template <int NB>
cudaError_t launch_mono(const KParams &K, size_t wbytes, int sms, int cap, cudaStream_t s)
{
    switch (K.reach) {
    case 3: return launch_mono_r<NB, 3>(K, wbytes, sms, cap, s);
    case 5: return launch_mono_r<NB, 5>(K, wbytes, sms, cap, s);
    case 7: return launch_mono_r<NB, 7>(K, wbytes, sms, cap, s);
    default: return cudaErrorInvalidValue;
    }
}

// the wide types' monopole kernel
template <typename T>
cudaError_t launch_mono_wide(const fmm_tree_s *t, const KParams &K, int sms, int cap, cudaStream_t s)
{
    MonoWParams P{};
    P.info = K.info;
    P.nbr = K.nbr;
    P.list = K.list;
    P.n_items = K.n_items;
    P.counter = K.counter;
    P.orbits = t->dev.orbits;
    for (int k = 0; k < 9; ++k) P.first[k] = t->orbit_first[k];
    P.coef = t->dev.orbit_coef;
    P.n_coef = int(t->orbit_coef.size());
    P.reach = (K.reach - 1) / 2;
    P.mass = K.mass;
    P.L = K.L;
    P.Lc = K.Lc;
    P.dL1 = K.dL1;
    // a CTA per node, or per plane of one while those do not fill the SMs
    const bool planes = K.n_items <= sms;
    const size_t bytes = mono_wide_smem<T>(P.reach, planes ? 1 : 4, P.n_coef);
    cudaError_t e = planes ? Kernels<T>::template mono_wide<1>(bytes) : Kernels<T>::template mono_wide<4>(bytes);
    if (e != cudaSuccess) return e;
    if (planes) {
        P.n_items = 4 * K.n_items;
        const int g = persistent_grid(mono_wide_kernel<T, 1>, bytes, P.n_items, sms, cap, 128);
        mono_wide_kernel<T, 1><<<g, 128, bytes, s>>>(P);
    } else {
        mono_wide_kernel<T, 4><<<std::min(P.n_items, sms), 512, bytes, s>>>(P);
    }
    return cudaGetLastError();
}

// the multipole launch of the wide types, PARTS items per sub-grid
template <typename T, int ORDER, int PARTS>
cudaError_t launch_mpw(KParams K, size_t bytes, int sms, int cap, cudaStream_t s)
{
    cudaError_t e = Kernels<T>::template mpw<ORDER, PARTS>(bytes);
    if (e != cudaSuccess) return e;
    K.n_items *= PARTS;
    const int g = persistent_grid(mpw_kernel<T, ORDER, PARTS>, bytes, K.n_items, sms, cap, kWideThreads);
    mpw_kernel<T, ORDER, PARTS><<<g, kWideThreads, bytes, s>>>(K);
    return cudaGetLastError();
}

// and of the mixed precision; window, compensation pairs and ring
template <int ORDER, int PARTS, bool AHEAD, int WARPS = 8>
cudaError_t launch_mp(KParams K, size_t wbytes, int sms, int cap, cudaStream_t s)
{
    constexpr int threads = 32 * WARPS;
    const size_t bytes = wbytes + size_t(kMpPairs) * 2 * threads * sizeof(float) +
                         size_t(threads) * (WARPS == 4 ? kMpDepth : 0) * 64;
    cudaError_t e = Kernels<float>::mp<ORDER, PARTS, AHEAD, WARPS>(bytes);
    if (e != cudaSuccess) return e;
    K.n_items *= PARTS;
    const int g = persistent_grid(mp_kernel<ORDER, PARTS, AHEAD, WARPS>, bytes, K.n_items, sms, cap, threads);
    mp_kernel<ORDER, PARTS, AHEAD, WARPS><<<g, threads, bytes, s>>>(K);
    return cudaGetLastError();
}
template <int ORDER>
cudaError_t launch_mp_split(KParams K, size_t wbytes, int sms, int cap, cudaStream_t s)
{
    const size_t bytes = wbytes + size_t(kMpPairs) * 2 * kSplitThreads * sizeof(float) +
                         size_t(kSplitThreads) * kSplitDepth * 64;
    cudaError_t e = Kernels<float>::mp_split<ORDER>(bytes);
    if (e != cudaSuccess) return e;
    K.n_items *= kSplitParts;
    const int g = persistent_grid(mp_split_kernel<ORDER>, bytes, K.n_items, sms, cap, kSplitThreads);
    mp_split_kernel<ORDER><<<g, kSplitThreads, bytes, s>>>(K);
    return cudaGetLastError();
}

template <typename T, int ORDER>
cudaError_t launch_all(const fmm_tree_s *t, void *L, float *Lc, double *dL1, cudaStream_t s,
                       int *n_launches, int parts)
{
    const Plan &Pl = t->plan;
    const DeviceTables &d = t->dev;
    KParams P{};
    P.info = d.info;
    P.nbr = d.nbr;
    P.stencil_f = reinterpret_cast<const float4 *>(d.stencil_f);
    P.coef = d.coef32;
    P.n_far = Pl.n_far[0];
    P.n_near = Pl.n_near[0];
    P.ent_stride = Pl.ent_stride;
    P.reach = Pl.reach;
    P.py = Pl.py;
    P.pz = Pl.pz;
    P.sub_stride = Pl.sub_stride;
    P.mass = d.mass;
    P.mp = d.mp;
    P.mp_limit = int(t->n_refined * 4 * NCELL * 4);
    P.L = L;
    P.Lc = Lc;
    P.dL1 = dL1;
    P.far_o2 = t->plan.far_o2;
    P.mx_targets = d.mx_targets;
    P.mx_pairs = d.mx_pairs;
    P.mono_woff = d.mono_woff;
    P.mono_woff16 = d.mono_woff16;
    const int cap = t->tuning.ctas_per_sm;
    const size_t wbytes = size_t(8) * Pl.sub_stride * sizeof(T);
    cudaError_t e;
    if (parts & M2L_RESET) {
        e = cudaMemsetAsync(d.counters, 0, 4 * sizeof(int32_t), s);
        if (e != cudaSuccess) return e;
    }
    const int sms = sm_count_of_current_device();
    int nl = 0;
    // M2L_MPX: the monopole<-multipole targets ride in the multipole launch
    // when there is one, else they get their own
    const bool mx_in_mp = (parts & M2L_MPX) && (parts & M2L_MP) && Pl.work_mp.count > 0;
    if ((parts & M2L_ROOT) && Pl.roots.count) {
        KParams R = P;
        R.list = d.lists + Pl.roots.off;
        R.n_items = int32_t(Pl.roots.count);
        timing_begin(t, FMM_K_ROOT, s);
        if constexpr (kF32<T>)
            root_kernel<ORDER><<<dim3(unsigned(Pl.roots.count), kRootGroups), kRootThreads, 0, s>>>(R);
        else
            rootw_kernel<T, ORDER><<<dim3(unsigned(Pl.roots.count), NCELL / kRootwTargets), kThreads, 0,
                                     s>>>(R);
        timing_end(t, s);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((parts & M2L_MP) && Pl.work_mp.count) {
        KParams K = P;
        K.list = d.lists + Pl.work_mp.off;
        K.n_items = int32_t(Pl.work_mp.count);
        K.counter = d.counters + Q_MP;
        if (mx_in_mp) {
            K.n_mx = int32_t(Pl.n_mx_targets);
            K.mx_counter = d.counters + Q_MX;
        }
        timing_begin(t, FMM_K_MULTIPOLE, s);
        if (kF32<T> && ORDER == 3 && t->tuning.mp_pair_targets) {
            // both target cells of a thread together (float only)
            const size_t b2 = wbytes + size_t(kMp2Pairs) * 2 * kThreads * sizeof(float);
            if ((e = Kernels<T>::mp2(b2)) != cudaSuccess) return e;
            int g = persistent_grid(mp2_kernel, b2, Pl.work_mp.count, sms, cap);
            mp2_kernel<<<g, kThreads, b2, s>>>(K);
        } else {
            const int mode = t->tuning.mp_items;
            const int64_t n = Pl.work_mp.count;
            if constexpr (kF32<T>) {
                // Few sub-grids, whose time is that of one warp's walk: pairs of
                // warps up to three pairs an SM, quarters of a sub-grid up to
                // two four-warp CTAs an SM, halves with the loads ahead up to
                // two such CTAs.  Steps of binaries, us, halves with the
                // loads ahead / this: 21 sub-grids 184 / 160, 41 204 / 177,
                // 72 272 / 257; above 76 quarters take two rounds (113:
                // 323 / 347).  Else half sub-grids per item where
                // whole ones would leave CTA slots idle or unbalanced (fewer
                // nodes than twice the slots).  Same bits throughout.
                if (mode == 0 && 16 * n <= 3 * int64_t(sms))
                    e = launch_mp_split<ORDER>(K, wbytes, sms, cap, s);
                else if (mode == 0 && 4 * n <= 2 * int64_t(sms))
                    e = launch_mp<ORDER, 4, false, 4>(K, wbytes, sms, cap, s);
                else if (mode == 0 && 2 * n <= 2 * int64_t(sms))
                    e = launch_mp<ORDER, 2, true>(K, wbytes, sms, cap, s);
                else if (mode == 2 || (mode == 0 && n < 2 * int64_t(cap > 0 && cap < 3 ? cap : 3) * sms))
                    e = launch_mp<ORDER, 2, false>(K, wbytes, sms, cap, s);
                else
                    e = launch_mp<ORDER, 1, false>(K, wbytes, sms, cap, s);
            } else {
                // halves and quarters of a sub-grid (mp_items 1 and 2; by
                // default quarters below eight nodes an SM, so that the last
                // items to run are short), and sixteenths where even quarters would not fill the SMs once
                // (whatever mp_items says: their sums round differently)
                const size_t fold = size_t(kWideThreads / 64) * kWideSums<ORDER> * 32 * sizeof(T);
                if (4 * n < sms)
                    e = launch_mpw<T, ORDER, 16>(K, std::max(wbytes, fold), sms, cap, s);
                else if (mode == 2 || (mode == 0 && n < 8 * int64_t(sms)))
                    e = launch_mpw<T, ORDER, 4>(K, wbytes, sms, cap, s);
                else
                    e = launch_mpw<T, ORDER, 2>(K, wbytes, sms, cap, s);
            }
            if (e != cudaSuccess) return e;
        }
        timing_end(t, s);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if ((parts & M2L_MONO) && Pl.work_mono.count) {
        KParams K = P;
        K.list = d.lists + Pl.work_mono.off;
        K.n_items = int32_t(Pl.work_mono.count);
        K.counter = d.counters + Q_MONO;
        timing_begin(t, FMM_K_MONOPOLE, s);
        if constexpr (kF32<T>) {
            int nb = t->tuning.mono_subgrids;
            if (nb != 1 && nb != 2 && nb != 4) nb = 2;
            // fewer sub-grids per pass where their windows do not fit
            const size_t smem_max = max_smem_optin_of_current_device();
            while (nb > 1 && mono_smem_bytes(nb, wbytes, Pl.ent_stride, false) > smem_max) nb /= 2;
            e = nb == 1 ? launch_mono<1>(K, wbytes, sms, cap, s)
                : nb == 2 ? launch_mono<2>(K, wbytes, sms, cap, s)
                          : launch_mono<4>(K, wbytes, sms, cap, s);
        } else {
            e = launch_mono_wide<T>(t, K, sms, cap, s);
        }
        timing_end(t, s);
        ++nl;
        if (e != cudaSuccess) return e;
    }
    if ((parts & (M2L_MX | M2L_MPX)) && !mx_in_mp && Pl.n_mx_targets) {
        KParams K = P;
        K.n_items = int32_t(Pl.n_mx_targets);
        const int64_t warps = (K.n_items + 31) / 32;
        int g = persistent_grid(mx_kernel<T, ORDER>, 0, (warps + kThreads / 32 - 1) / (kThreads / 32), sms,
                                cap);
        timing_begin(t, FMM_K_MONO_MULTI, s);
        mx_kernel<T, ORDER><<<g, kThreads, 0, s>>>(K);
        timing_end(t, s);
        ++nl;
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (n_launches) *n_launches = nl;
    return cudaSuccess;
}

template <typename T>
void launch_pack_t(const fmm_tree_s *t, const double *M, const double *com, cudaStream_t s,
                   const int32_t *nodes, int64_t count)
{
    const auto &c = t->cfg;
    pack_kernel<T><<<unsigned(count), 512, 0, s>>>(t->dev.info, nodes, t->dev.levels, M, com,
                                                   static_cast<T *>(t->dev.mass),
                                                   static_cast<T *>(t->dev.mp), c.box_lo[0],
                                                   c.box_lo[1], c.box_lo[2]);
}

}  // namespace

cudaError_t launch_pack(const fmm_tree_s *t, const double *M, const double *com, cudaStream_t s,
                        int which)
{
    const int32_t *nodes = nullptr;
    int64_t count = t->n;
    if (which == PACK_LEAVES) {
        nodes = t->dev.lists + t->plan.leaves.off;
        count = t->plan.leaves.count;
    } else if (which == PACK_REFINED) {
        nodes = t->dev.lists + t->plan.refined.off;
        count = t->plan.refined.count;
    }
    if (count == 0) return cudaSuccess;
    switch (t->cfg.precision) {
    case FMM_MIXED: launch_pack_t<float>(t, M, com, s, nodes, count); break;
    case FMM_DFLOAT: launch_pack_t<dfloat>(t, M, com, s, nodes, count); break;
    default: launch_pack_t<double>(t, M, com, s, nodes, count); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_m2l(const fmm_tree_s *t, void *L, float *Lc, double *dL1, cudaStream_t s,
                       int *n_launches, int parts)
{
    const bool o2 = t->cfg.order == 2;
    switch (t->cfg.precision) {
    case FMM_MIXED:
        return o2 ? launch_all<float, 2>(t, L, Lc, dL1, s, n_launches, parts)
                  : launch_all<float, 3>(t, L, Lc, dL1, s, n_launches, parts);
    case FMM_DFLOAT:
        return o2 ? launch_all<dfloat, 2>(t, L, Lc, dL1, s, n_launches, parts)
                  : launch_all<dfloat, 3>(t, L, Lc, dL1, s, n_launches, parts);
    default:
        return o2 ? launch_all<double, 2>(t, L, Lc, dL1, s, n_launches, parts)
                  : launch_all<double, 3>(t, L, Lc, dL1, s, n_launches, parts);
    }
}

}  // namespace fmm
