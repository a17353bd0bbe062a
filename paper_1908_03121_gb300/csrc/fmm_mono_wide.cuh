// Monopole<-monopole in the wide element types (double, double-float).
//
// Leaf targets and leaf sources: a convolution of the masses with weights
// w_c(o), c = 0 (L0, even in every axis) or an axis (L1, odd in that axis).
// Both types are bound by their arithmetic pipe, so the sum is taken in the
// basis in which the stencil's reflections are diagonal, with an eighth of
// the products:
//   - the stencil of the opening rule is all children s of the near parents:
//     seen from child p of block C (2 x 2 x 2 cells), child s of block C + d
//     lies at o = 2 d + s - p, for every d that is not well separated;
//   - sources and targets go through the Hadamard transform of their block's
//     eight children, m^_b = sum_s (-1)^(b.s) m_s and out_p = sum_a (-1)^(a.p)
//     O_a, which turns the 8 x 8 weights of one d into
//       K_ab(d) = (1/64) sum_ps (-1)^(a.p + b.s) w_c(2 d + s - p),
//     even or odd in each axis of d (odd iff a, b and e_c add up to an odd bit
//     there: q = a xor b xor e_c);
//   - so the blocks d that differ in signs only are first combined,
//       S_b^q(C) = sum_signs (product of the signs of q's axes) m^_b(C + d),
//     and O_a += K_ab(|d|) S_b^q: one product per (b, q, c), where the direct
//     form has one per (p, s, c) and sign.
//   - only the own block (d = 0) is summed directly, cell by cell: in the
//     transformed basis a cell's own mass would enter its sums and cancel to
//     rounding of that mass alone, far above the field of a thin surrounding (a
//     dense cell in a floor of 1e-10: 9e-9 of g in FP64).  A heavier cell of
//     another block attracts the target by as much as its roundings scale with.
// theta = 0.5: 1024 products, 480 additions, 192 + 320 for the transforms and 152
// products in the own block per block of eight cells, against 8416 products
// (direct form).  A level-6 binary
// (4572 leaf nodes), whole step: FP64 24.1 -> 20.9 ms (this kernel 4.4 -> 1.2),
// double-float 5.43 -> 4.79 ms; 8 leaf nodes in FP64, step 318 -> 207 us.  (The
// own block's products, spread over all threads, cost 0.11 and 0.04 ms of a level-6
// step, 1 us of 8 leaf nodes'; by the 128 threads of the exchange 0.13, 0.07 and 2.)
// A thread has one target block and one b (the same for a whole warp, so the
// weights are broadcasts); its 32 sums A[q][c] belong to a = q xor b xor e_c and
// meet those of the other b at the end, through shared memory, in a fixed
// order.  A CTA takes PLANES of the four planes of blocks of a leaf node: all
// four with 16 warps, one CTA per SM, or one with four warps where there are
// few leaf nodes.  Same bits.  (A 9-sub-grid step in FP64, its root beside this
// kernel: 172 -> 148 us.)
#pragma once

#include "fmm_internal.h"
#include "fmm_tensor.cuh"

namespace fmm {

namespace {

struct MonoWParams {
    const NodeInfo *info;
    const int32_t *nbr;
    const int32_t *list;
    int32_t n_items;
    int32_t *counter;
    const int4 *orbits;          // [n] (dx, dy, dz >= 0, mask of nonzero axes), by mask
    int first[9];                // orbits of mask k: first[k] .. first[k + 1]
    const void *coef;            // [orbit][b][q in mask][c]; the last eight: [2][4] within a block
    int n_coef;                  // values
    int reach;                   // in blocks
    const void *mass;
    void *L;
    float *Lc;
    double *dL1;
};

// window of (4 + 2 R)^2 (planes + 2 R) blocks; the row pitch 12 puts the 16
// (x, y) lanes of a half warp on distinct banks for 8-byte elements
constexpr int kMonoWPitch = 12;
__host__ __device__ constexpr int mono_wide_window(int reach, int planes)
{
    return kMonoWPitch * (4 + 2 * reach) * (planes + 2 * reach);
}

// shared memory: the window (later the exchange buffer, two components of 8 sums
// and one own-block value of every thread) and the weights
template <typename T>
size_t mono_wide_smem(int reach, int planes, int n_coef)
{
    const size_t window = size_t(8) * mono_wide_window(reach, planes), fold = size_t(2) * 9 * 128 * planes;
    return ((window > fold ? window : fold) + size_t(n_coef)) * sizeof(T);
}

// one orbit of blocks with nonzero axes MASK into the thread's sums
template <typename T, int MASK>
__device__ __forceinline__ void mono_wide_orbit(const T *W, int dx, int dy, int dz, const T *coef,
                                                T (&A)[8][4])
{
    T v[8];
    // the blocks of all sign combinations (bit set: the negative side)
#pragma unroll
    for (int s = 0; s < 8; ++s)
        if ((s & ~MASK) == 0) v[s] = W[((s & 1) ? -dx : dx) + ((s & 2) ? -dy : dy) + ((s & 4) ? -dz : dz)];
    // sums and differences per axis: v[q] becomes S^q
#pragma unroll
    for (int ax = 1; ax < 8; ax <<= 1) {
        if (!(MASK & ax)) continue;
#pragma unroll
        for (int s = 0; s < 8; ++s) {
            if ((s & ~MASK) || (s & ax)) continue;
            const T a = v[s], b = v[s | ax];
            v[s] = add_u(a, b);
            v[s | ax] = add_u(a, -b);
        }
    }
    int at = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        if (q & ~MASK) continue;
        T c[4];
        load4_shared<T>(coef + at, c);
        at += 4;
#pragma unroll
        for (int k = 0; k < 4; ++k) A[q][k] = fmadd_u(c[k], v[q], A[q][k]);
    }
}

template <typename T, int MASK>
__device__ __forceinline__ void mono_wide_orbits(const MonoWParams &P, const T *W, int pz, int b,
                                                 const T *&coef, T (&A)[8][4])
{
    constexpr int nq = 1 << (((MASK >> 0) & 1) + ((MASK >> 1) & 1) + ((MASK >> 2) & 1));
    for (int i = P.first[MASK]; i < P.first[MASK + 1]; ++i) {
        const int4 o = __ldg(P.orbits + i);
        mono_wide_orbit<T, MASK>(W, o.x, kMonoWPitch * o.y, pz * o.z, coef + b * nq * 4, A);
        coef += 8 * nq * 4;
    }
    // canonical form of the sums (double-float; at most 19 orbits of a mask)
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) A[q][k] = renorm(A[q][k]);
}

// the own block's terms of one component for target child p, from the masses
// m[x] of its children p xor x: EC = 0 for L0, else the axis's bit (a first-order
// weight is nonzero between cells apart in that axis only, and its sign is the
// target's side of it)
template <typename T, int EC>
__device__ __forceinline__ T mono_wide_own(const T m[8], const T *near, int p)
{
    T v = T(0);
#pragma unroll
    for (int x = 1; x < 8; ++x)
        if (EC == 0 || (x & EC))
            v = fmadd_u(near[(EC ? 4 : 0) + (x & 1) + ((x >> 1) & 1) + (x >> 2) - 1], m[x], v);
    v = renorm(v);
    return (p & EC) ? -v : v;
}

template <typename T, int PLANES>
__global__ void __launch_bounds__(128 * PLANES, PLANES == 4 ? 1 : 4) mono_wide_kernel(MonoWParams P)
{
    constexpr int blocks = 16 * PLANES;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_nbr[27], s_item;
    const int R = P.reach, E = 4 + 2 * R, EZ = PLANES + 2 * R, pz = kMonoWPitch * E;
    const int plane = pz * EZ;                           // blocks of one b
    const int sums = 2 * 8 * 8 * blocks, fold = sums + 2 * 8 * blocks;
    T *W = reinterpret_cast<T *>(smem_raw);
    T *s_coef = W + (8 * plane > fold ? 8 * plane : fold);
    const T *mass = static_cast<const T *>(P.mass);
    for (int i = threadIdx.x; i < P.n_coef; i += blockDim.x)
        s_coef[i] = ldg_t(static_cast<const T *>(P.coef) + i);
    const int b = threadIdx.x / blocks, block = threadIdx.x % blocks;   // target block x + 4 y + 16 z
    const int tx = block & 3, ty = (block >> 2) & 3, tz = block >> 4;
    for (;;) {
        const int item = pull_item(P.counter, &s_item);
        if (item >= P.n_items) break;
        const int node = P.list[item / (4 / PLANES)];
        const int z0 = item % (4 / PLANES) * PLANES;           // the CTA's first plane
        // leaf neighbours (-1: absent or refined)
        if (threadIdx.x < 27) {
            const int nb = P.nbr[node * 27 + threadIdx.x];
            s_nbr[threadIdx.x] = nb >= 0 && P.info[nb].leaf_row >= 0 ? nb : -1;
        }
        __syncthreads();
        // the window's masses, child s of block u to plane s (the packed mass
        // array has a node's child-s cells contiguous)
        for (int i = threadIdx.x; i < E * E * EZ; i += blockDim.x) {
            const int ux = i % E, uy = (i / E) % E, uz = i / (E * E);
            const int bx = ux - R + 4, by = uy - R + 4, bz = uz - R + z0 + 4; // >= 1
            const int nb = s_nbr[(bx >> 2) + 3 * (by >> 2) + 9 * (bz >> 2)];
            const int src = (bx & 3) + 4 * (by & 3) + 16 * (bz & 3);
            const T *from = nb >= 0 ? mass + size_t(nb) * NCELL + src : mass;
            T *to = W + ux + kMonoWPitch * uy + pz * uz;
#pragma unroll
            for (int s = 0; s < 8; ++s) cp_async_elem<T>(to + s * plane, from + (nb >= 0 ? 64 * s : 0), nb >= 0);
        }
        cp_async_commit();
        cp_async_wait_all();
        // (each thread transforms the blocks that it staged itself)
        for (int i = threadIdx.x; i < E * E * EZ; i += blockDim.x) {
            T *at = W + i % E + kMonoWPitch * ((i / E) % E) + pz * (i / (E * E));
            T m[8];
#pragma unroll
            for (int s = 0; s < 8; ++s) m[s] = at[s * plane];
#pragma unroll
            for (int ax = 1; ax < 8; ax <<= 1)
#pragma unroll
                for (int s = 0; s < 8; ++s) {
                    if (s & ax) continue;
                    const T u = m[s], v = m[s | ax];
                    m[s] = u + v;
                    m[s | ax] = u - v;
                }
#pragma unroll
            for (int s = 0; s < 8; ++s) at[s * plane] = m[s];
        }
        __syncthreads();
        T A[8][4];
#pragma unroll
        for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int k = 0; k < 4; ++k) A[q][k] = T(0);
        const T *own = W + b * plane + (tx + R) + kMonoWPitch * (ty + R) + pz * (tz + R);
        const T *coef = s_coef;
        mono_wide_orbits<T, 1>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 2>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 3>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 4>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 5>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 6>(P, own, pz, b, coef, A);
        mono_wide_orbits<T, 7>(P, own, pz, b, coef, A);
        // O_a[c] = sum_b A^b[a xor b xor e_c][c], then out_p = sum_a (-1)^(a.p) O_a:
        // components 0-1, then 2-3, one thread per (component, target block)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            // the own block's terms for child b of this thread's block
            T m[8];
            const T *at = mass + size_t(node) * NCELL + tx + 4 * ty + 16 * (z0 + tz);
#pragma unroll
            for (int x = 1; x < 8; ++x) m[x] = ldg_t(at + 64 * (b ^ x));
            const T *near = s_coef + P.n_coef - 8;
            __syncthreads();                           // the window (the first half) is done with
            W[sums + b * blocks + block] = half ? mono_wide_own<T, 2>(m, near, b) : mono_wide_own<T, 0>(m, near, b);
            W[sums + (8 + b) * blocks + block] = half ? mono_wide_own<T, 4>(m, near, b) : mono_wide_own<T, 1>(m, near, b);
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
                for (int q = 0; q < 8; ++q) W[((k * 8 + b) * 8 + q) * blocks + block] = A[q][2 * half + k];
            __syncthreads();
            if (threadIdx.x < 2 * blocks) {
                const int k = threadIdx.x / blocks, t = threadIdx.x % blocks;
                const int c = 2 * half + k;
                const int ec = c == 0 ? 0 : 1 << (c - 1);
                T o[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    T v = W[(k * 64 + (a ^ ec)) * blocks + t];
#pragma unroll
                    for (int s = 1; s < 8; ++s) v += W[((k * 8 + s) * 8 + (a ^ s ^ ec)) * blocks + t];
                    o[a] = v;
                }
#pragma unroll
                for (int ax = 1; ax < 8; ax <<= 1)
#pragma unroll
                    for (int a = 0; a < 8; ++a) {
                        if (a & ax) continue;
                        const T u = o[a], v = o[a | ax];
                        o[a] = u + v;
                        o[a | ax] = u - v;
                    }
#pragma unroll
                for (int p = 0; p < 8; ++p) o[p] += W[sums + (8 * k + p) * blocks + t];
                const int cell = 2 * (t & 3) + 16 * ((t >> 2) & 3) + 128 * (z0 + (t >> 4));
#pragma unroll
                for (int p = 0; p < 8; ++p)
                    store_L<T>(P, node, c, cell + (p & 1) + 8 * ((p >> 1) & 1) + 64 * (p >> 2), o[p], T(0));
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) __stcs(P.dL1 + (size_t(node) * 3 + i) * NCELL + 128 * z0 + threadIdx.x, 0.0);
        __syncthreads();
    }
}

}  // namespace

}  // namespace fmm
