// Self-consistent-field (SCF) initial models: the second caller of the
// gravity solve.  The paper builds its V1309 initial model with Octo-Tiger's
// SCF module, which iterates the FMM solve (Sec. 3, Sec. 4.2; the method is
// Hachisu's 1986 self-consistent field for rotating stars and binaries).
//
// fmm_scf_update performs one iteration's density update after a solve of
// the same tree, for polytropes P = K rho^(1 + 1/n) in synchronous rotation
// about the z axis through the centre of mass:
//   H = C_i - Phi + Omega^2 w^2 / 2   (the enthalpy (n + 1) K_i rho^(1/n)
//                                     inside star i, w the axis distance),
//   Omega^2, C_1, C_2 from H = 0 at surface points A, B (star 1) and C
//   (star 2),  rho' = max(rho_floor, rho_max,i (H / H_max,i)^n) where H > 0.
// The per-cell work (centre of mass, H and its per-star maximum, the new
// density) runs in three kernels over the leaf nodes; the last CTA of the first
// two to finish combines the nodes' values in a fixed order and writes them
// into page-locked host memory (with the potential at the three surface
// cells), from which the host forms the few scalars of the iteration in FP64.
// An update of 512 leaf nodes, with its solve: 355 -> 293 us against copies of
// every node's partial sums through pageable memory and full shuffle trees of
// FP64 adds per node.  FP64 operations bound the three kernels, so nodes that
// neither star reaches are sorted out in float, a thread's two cells share what
// x and y set, and the mass sums are taken in cell indices: 273 -> 257 us.
#include <cmath>
#include <string>

#include "fmm_chain.cuh"
#include "fmm_convert.cuh"
#include "fmm_internal.h"

namespace fmm {
namespace {

constexpr int kScfThreads = 256;       // 2 cells per thread, four planes apart
static_assert(NCELL == 2 * kScfThreads, "two cells per thread");

struct ScfGeo {
    double lo[3];
    double size;
};

// a small whole number as a double, on the integer pipe
__device__ __forceinline__ double whole(int i) { return f2d_bits(float(i)); }

// centre of a cell along one axis: node index i, cell index k
__device__ __forceinline__ double centre_of(double lo, int i, int k, double h)
{
    return lo + (8.0 * i + whole(k) + 0.5) * h;
}

// fixed-order sum or maximum of every component k of the 256 threads' v[k]; the
// results in threads 0 .. NV - 1.  Sixteen threads per component combine
// sixteen values each, then one the sixteen: 31 dependent FP64 operations,
// where a shuffle tree has all eight warps at work on each of its levels.
template <int NV, bool MAX>
__device__ __forceinline__ double block_combine(const double v[NV])
{
    __shared__ double sh[NV][kScfThreads + kScfThreads / 16];
    __shared__ double part[NV][16];
    auto both = [](double a, double b) { return MAX ? fmax(a, b) : a + b; };
#pragma unroll
    for (int k = 0; k < NV; ++k) sh[k][threadIdx.x + threadIdx.x / 16] = v[k];
    __syncthreads();
    if (threadIdx.x < 16 * NV) {
        const int k = threadIdx.x >> 4, q = threadIdx.x & 15;
        double t = sh[k][17 * q];
#pragma unroll
        for (int i = 1; i < 16; ++i) t = both(t, sh[k][17 * q + i]);
        part[k][q] = t;
    }
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < NV) {
        t = part[threadIdx.x][0];
#pragma unroll
        for (int q = 1; q < 16; ++q) t = both(t, part[threadIdx.x][q]);
    }
    return t;
}

// the node's value of component k (threads 0 .. NV - 1) into its row; in the
// last CTA of the launch, true, with the rows' combined values in threads
// 0 .. NV - 1 of `all`
template <int NV, bool MAX>
__device__ __forceinline__ bool combine_nodes(double mine, int row, double *partials, int32_t *arrived,
                                              double &all)
{
    __shared__ int s_last;
    if (threadIdx.x < NV) {
        partials[size_t(row) * 8 + threadIdx.x] = mine;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(arrived, 1) == int(gridDim.x) - 1;
    __syncthreads();
    if (!s_last) return false;
    __threadfence();
    double v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = MAX ? -1e300 : 0.0;
    for (int i = threadIdx.x; i < int(gridDim.x); i += kScfThreads)
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const double o = load_cg(partials + size_t(i) * 8 + k);     // other CTAs' rows
            v[k] = MAX ? fmax(v[k], o) : v[k] + o;
        }
    all = block_combine<NV, MAX>(v);
    if (threadIdx.x == 0) *arrived = 0;
    return true;
}

// the potential's address at the three surface cells
struct ScfPoints {
    const double *phi[3];
};

// sum m, sum m x, sum m y, sum m z (m = rho h^3) over the leaf nodes into
// host[0..3], the potentials at the points into host[4..6]
__global__ void __launch_bounds__(kScfThreads) scf_com_kernel(const NodeInfo *__restrict__ info,
                                                               const int32_t *__restrict__ leaves,
                                                               const double *__restrict__ levels,
                                                               const double *__restrict__ rho,
                                                               double *__restrict__ partials,
                                                               int32_t *__restrict__ arrived, ScfGeo g,
                                                               ScfPoints points, double *host)
{
    // density sums in cell indices; the node's scale and corner at the end
    const NodeInfo ni = info[leaves[blockIdx.x]];
    const double *r = rho + size_t(ni.leaf_row) * NCELL + threadIdx.x;
    const double r0 = r[0], r1 = r[kScfThreads], both = r0 + r1;
    const int c = threadIdx.x;
    const double v[4] = {both, both * whole(c & 7), both * whole((c >> 3) & 7),
                         fma(r0, whole(c >> 6), r1 * whole((c >> 6) + 4))};
    double mine = block_combine<4, false>(v);
    if (threadIdx.x < 32) {
        const double sum = __shfl_sync(0xffffffffu, mine, 0);
        const double h = levels[ni.level * LEVEL_FIELDS + LV_H], h3 = levels[ni.level * LEVEL_FIELDS + LV_H3];
        if (threadIdx.x > 0 && threadIdx.x < 4) {
            const int a = threadIdx.x;
            const double corner = a == 1   ? centre_of(g.lo[0], ni.ix, 0, h)
                                  : a == 2 ? centre_of(g.lo[1], ni.iy, 0, h)
                                           : centre_of(g.lo[2], ni.iz, 0, h);
            mine = fma(corner, sum, h * mine);
        }
        mine *= h3;
    }
    double all;
    if (!combine_nodes<4, false>(mine, ni.leaf_row, partials, arrived, all)) return;
    if (threadIdx.x < 4) host[threadIdx.x] = all;
    else if (threadIdx.x < 7) host[threadIdx.x] = *points.phi[threadIdx.x - 4];
}

struct ScfStars {
    double omega2, C[2], com[2], x_split;
    double centre[2][3], r2lim[2];
    int live[2];                         // star i exists (rho_max > 0)
    float box_centre[2][3], box_reach[2];  // in box widths; the reach rounded up
};

// whether any cell of the node can lie within a star's reach: the distance from
// the star's centre to the box of the node's cell centres, in float, against
// the reach with a margin far above float's rounding.  Most nodes lie in
// neither star and take none of the FP64 operations per cell, which bound both
// kernels
__device__ __forceinline__ bool near_star(const NodeInfo &ni, const ScfStars &s)
{
    const int at[3] = {ni.ix, ni.iy, ni.iz};
    const float w = exp2f(float(1 - ni.level));
    bool near = false;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        float d2 = 0.f;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float lo = (float(at[a]) + 0.0625f) * w, hi = (float(at[a]) + 0.9375f) * w;
            const float d = fmaxf(fmaxf(lo - s.box_centre[i][a], s.box_centre[i][a] - hi), 0.f);
            d2 = fmaf(d, d, d2);
        }
        near = near || (s.live[i] && !(d2 > s.box_reach[i] * s.box_reach[i]));
    }
    return near;
}

// a thread's two cells (x, y alike): the star they may belong to, 0 or 1, or -1,
// and the parts of the distance and the enthalpy that x and y set
struct ScfColumn {
    int star;
    double d2, rot, h;
    __device__ __forceinline__ ScfColumn(const NodeInfo &ni, double h_, const ScfGeo &g, const ScfStars &s)
        : h(h_)
    {
        const int c = threadIdx.x;
        const double x = centre_of(g.lo[0], ni.ix, c & 7, h), y = centre_of(g.lo[1], ni.iy, (c >> 3) & 7, h);
        star = x < s.x_split ? 0 : 1;
        const double dx = x - s.centre[star][0], dy = y - s.centre[star][1];
        d2 = fma(dy, dy, fma(dx, dx, 0.0));
        if (!s.live[star]) star = -1;
        const double wx = x - s.com[0], wy = y - s.com[1];
        rot = 0.5 * s.omega2 * fma(wx, wx, wy * wy);
    }
    // whether cell threadIdx.x + 256 j is inside the star
    __device__ __forceinline__ bool inside(const NodeInfo &ni, const ScfGeo &g, const ScfStars &s, int j) const
    {
        if (star < 0) return false;
        const double dz = centre_of(g.lo[2], ni.iz, (int(threadIdx.x) >> 6) + 4 * j, h) - s.centre[star][2];
        return fma(dz, dz, d2) < s.r2lim[star];
    }
    __device__ __forceinline__ double enthalpy(double phi, const ScfStars &s) const
    {
        return s.C[star] - phi + rot;
    }
};

// the largest H of each star's cells into host[0..1]
__global__ void __launch_bounds__(kScfThreads) scf_hmax_kernel(const NodeInfo *__restrict__ info,
                                                                const int32_t *__restrict__ leaves,
                                                                const double *__restrict__ levels,
                                                                const double *__restrict__ phi,
                                                                double *__restrict__ partials,
                                                                int32_t *__restrict__ arrived, ScfGeo g,
                                                                ScfStars s, double *host)
{
    const NodeInfo ni = info[leaves[blockIdx.x]];
    double mine = -1e300;
    if (near_star(ni, s)) {              // (the same for the whole CTA)
        const ScfColumn col(ni, levels[ni.level * LEVEL_FIELDS + LV_H], g, s);
        const double *at = phi + size_t(ni.leaf_row) * NCELL + threadIdx.x;
        double m = -1e300;
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (col.inside(ni, g, s, j)) m = fmax(m, col.enthalpy(at[j * kScfThreads], s));
        const double v[2] = {col.star == 0 ? m : -1e300, col.star == 1 ? m : -1e300};
        mine = block_combine<2, true>(v);
    }
    double all;
    if (!combine_nodes<2, true>(mine, ni.leaf_row, partials, arrived, all)) return;
    if (threadIdx.x < 2) host[threadIdx.x] = all;
}

// u^n, u > 0; half: 2 n where that is a whole number up to 16 (the usual
// indices: products and a square root, a fifth of pow's FP64 operations).  What
// each rounding leaves out is carried along, so that the result is within one
// unit in the last place, as pow's is (2.6 without, at n = 7.5)
__device__ __forceinline__ double power(double u, double n, int half)
{
    if (half == 0) return pow(u, n);
    double r = 1.0, e = 0.0;             // the power so far is r + e
    if (half & 1) {
        r = sqrt(u);
        const float rf = d2f_trunc(r);   // (e to a float's bits)
        if (rf > 0.f) e = fma(-r, r, u) * f2d_bits(0.5f / rf);
    }
    for (int k = half >> 1; k > 0; --k) {
        const double p = r * u;
        e = fma(e, u, fma(r, u, -p));
        r = p;
    }
    return r + e;
}

// the new density: max(floor, rho_max,i (H / H_max,i)^n) inside star i where
// H > 0, the floor elsewhere (continuous in H: a cell whose H is zero to
// rounding takes the floor on either side of zero)
__global__ void __launch_bounds__(kScfThreads) scf_density_kernel(
    const NodeInfo *__restrict__ info, const int32_t *__restrict__ leaves,
    const double *__restrict__ levels, const double *__restrict__ phi, double *__restrict__ rho_out,
    ScfGeo g, ScfStars s, double n, int half, double rho_max0, double rho_max1, double ih0,
    double ih1, double floor_value)
{
    const NodeInfo ni = info[leaves[blockIdx.x]];
    const size_t at = size_t(ni.leaf_row) * NCELL + threadIdx.x;
    double r[2] = {floor_value, floor_value};
    if (near_star(ni, s)) {
        const ScfColumn col(ni, levels[ni.level * LEVEL_FIELDS + LV_H], g, s);
#pragma unroll
        for (int j = 0; j < 2; ++j)
            if (col.inside(ni, g, s, j)) {
                const double H = col.enthalpy(phi[at + j * kScfThreads], s);
                if (H > 0.0)
                    r[j] = fmax(floor_value, (col.star ? rho_max1 : rho_max0) *
                                                 power(H * (col.star ? ih1 : ih0), n, half));
            }
    }
    rho_out[at] = r[0];
    rho_out[at + kScfThreads] = r[1];
}

int scf_fail(int code, const std::string &msg)
{
    record_error("fmm_scf_update: " + msg);
    return code;
}

// leaf row, cell and cell centre of the leaf cell containing a point (false
// if none)
bool find_cell(const fmm_tree_s *t, const double p[3], int64_t &row, int &cell, double centre[3])
{
    // the point in units of the domain, and from the root down the child that
    // holds it
    const double *lo = t->cfg.box_lo;
    double f[3];
    for (int a = 0; a < 3; ++a) {
        f[a] = (p[a] - lo[a]) / t->cfg.box_size;
        if (!(f[a] >= 0.0 && f[a] < 1.0)) return false;
    }
    int64_t node = t->lists[size_t(t->plan.roots.off)];
    for (double n = 2.0; t->info[size_t(node)].leaf_row < 0; n *= 2.0) {
        int k = 0;
        for (int a = 0; a < 3; ++a) k |= (int64_t(std::floor(f[a] * n)) & 1) << a;
        node = t->children[size_t(node) * 8 + k];
    }
    const NodeInfo &ni = t->info[size_t(node)];
    const double n = std::ldexp(1.0, ni.level - 1);
    const int32_t ij[3] = {ni.ix, ni.iy, ni.iz};
    const double h = t->cfg.box_size / (8.0 * n);
    int k[3];
    for (int a = 0; a < 3; ++a) {
        k[a] = int(std::floor((f[a] * n - ij[a]) * 8.0));
        centre[a] = lo[a] + (8.0 * ij[a] + k[a] + 0.5) * h;
    }
    row = ni.leaf_row;
    cell = k[0] + 8 * k[1] + 64 * k[2];
    return true;
}

}  // namespace
}  // namespace fmm

extern "C" int fmm_scf_update(fmm_tree_t t, const fmm_scf_params *p, const double *phi,
                              const double *rho, double *rho_out, fmm_scf_result *out,
                              fmm_stream_t stream)
{
    using namespace fmm;
    if (!t || !p || !phi || !rho || !rho_out || !out) return scf_fail(FMM_ERR_INVALID_ARG, "NULL argument");
    if (t->host_only) return scf_fail(FMM_ERR_INVALID_ARG, "tree was planned with FMM_FLAG_HOST_ONLY");
    if (t->n_trees != 1) return scf_fail(FMM_ERR_INVALID_ARG, "the tree must hold a single tree");
    if (!(p->n > 0.0) || !(p->rho_max[0] > 0.0) || !(p->rho_max[1] >= 0.0) ||
        !(p->rho_floor >= 0.0) || !(p->r_lim[0] > 0.0) ||
        !(p->r_lim[1] >= 0.0) || (p->rho_max[1] > 0.0 && !(p->r_lim[1] > 0.0)))
        return scf_fail(FMM_ERR_INVALID_ARG, "n, rho_max[0] and r_lim[0] must be positive, "
                                             "rho_max[1], r_lim[1] and rho_floor not negative");
    const int64_t nl = t->n_leaf;
    // the surface conditions hold at the centres of the cells containing the
    // points, where the potential is known
    int64_t row[3] = {0, 0, 0};       // (a point that is not used: the first leaf cell)
    int cell[3] = {0, 0, 0};
    double ctr[3][3] = {{0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}, {0.0, 0.0, 0.0}};
    const double *pts[3] = {p->point_a, p->point_b, p->point_c};
    for (int k = 0; k < 3; ++k) {
        if (k == 1 && !p->rotate) continue;
        if (k == 2 && p->rho_max[1] <= 0.0) continue;
        if (!find_cell(t, pts[k], row[k], cell[k], ctr[k]))
            return scf_fail(FMM_ERR_INVALID_ARG, "a surface point lies outside every leaf node");
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int32_t *leaves = t->dev.lists + t->plan.leaves.off;
    const ScfGeo g{{t->cfg.box_lo[0], t->cfg.box_lo[1], t->cfg.box_lo[2]}, t->cfg.box_size};
    // 1. centre of mass; the potential at the surface cells
    ScfPoints points{};
    for (int k = 0; k < 3; ++k) points.phi[k] = phi + row[k] * NCELL + cell[k];
    scf_com_kernel<<<unsigned(nl), kScfThreads, 0, s>>>(t->dev.info, leaves, t->dev.levels, rho,
                                                         t->dev.partials, t->dev.reduce_arrived, g,
                                                         points, t->scf_host);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return scf_fail(FMM_ERR_CUDA, cudaGetErrorString(e));
    const double msum = t->scf_host[0], mx = t->scf_host[1], my = t->scf_host[2], mz = t->scf_host[3];
    const double phis[3] = {t->scf_host[4], t->scf_host[5], t->scf_host[6]};
    if (!(msum > 0.0)) return scf_fail(FMM_ERR_INVALID_ARG, "the density has no positive mass");
    ScfStars st{};
    st.com[0] = mx / msum;
    st.com[1] = my / msum;
    auto w2 = [&](const double *q) {
        const double dx = q[0] - st.com[0], dy = q[1] - st.com[1];
        return dx * dx + dy * dy;
    };
    // 2. the iteration's scalars from H = 0 at the surface points
    st.omega2 = 0.0;
    if (p->rotate) {
        const double den = w2(ctr[0]) - w2(ctr[1]);
        if (den == 0.0) return scf_fail(FMM_ERR_INVALID_ARG, "points A and B are equally far from the axis");
        st.omega2 = 2.0 * (phis[0] - phis[1]) / den;
    }
    st.C[0] = phis[0] - 0.5 * st.omega2 * w2(ctr[0]);
    st.C[1] = p->rho_max[1] > 0.0 ? phis[2] - 0.5 * st.omega2 * w2(ctr[2]) : 0.0;
    st.x_split = p->x_split;
    for (int i = 0; i < 2; ++i) {
        for (int a = 0; a < 3; ++a) st.centre[i][a] = p->centre[i][a];
        st.r2lim[i] = p->r_lim[i] * p->r_lim[i];
        st.live[i] = p->rho_max[i] > 0.0;
        double far = 1.0;
        for (int a = 0; a < 3; ++a) {
            const double c = (p->centre[i][a] - g.lo[a]) / g.size;
            st.box_centre[i][a] = float(c);
            far += std::abs(c);
        }
        st.box_reach[i] = float(p->r_lim[i] / g.size + 1e-5 * far);
    }
    // 3. each star's largest enthalpy
    scf_hmax_kernel<<<unsigned(nl), kScfThreads, 0, s>>>(t->dev.info, leaves, t->dev.levels, phi,
                                                          t->dev.partials, t->dev.reduce_arrived, g, st,
                                                          t->scf_host);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return scf_fail(FMM_ERR_CUDA, cudaGetErrorString(e));
    const double hmax[2] = {t->scf_host[0], t->scf_host[1]};
    for (int i = 0; i < 2; ++i)
        if (st.live[i] && !(hmax[i] > 0.0))
            return scf_fail(FMM_ERR_INVALID_ARG, "a star has no cell with positive enthalpy");
    // 4. the new density
    const int half = 2.0 * p->n <= 16.0 && 2.0 * p->n == std::floor(2.0 * p->n) ? int(2.0 * p->n) : 0;
    scf_density_kernel<<<unsigned(nl), kScfThreads, 0, s>>>(
        t->dev.info, leaves, t->dev.levels, phi, rho_out, g, st, p->n, half, p->rho_max[0],
        p->rho_max[1], 1.0 / hmax[0], st.live[1] ? 1.0 / hmax[1] : 0.0, p->rho_floor);
    e = cudaGetLastError();
    if (e != cudaSuccess) return scf_fail(FMM_ERR_CUDA, cudaGetErrorString(e));
    out->omega2 = st.omega2;
    out->C[0] = st.C[0];
    out->C[1] = st.C[1];
    out->com[0] = st.com[0];
    out->com[1] = st.com[1];
    out->com[2] = mz / msum;
    out->H_max[0] = hmax[0];
    out->H_max[1] = st.live[1] ? hmax[1] : 0.0;
    out->phi_points[0] = phis[0];
    out->phi_points[1] = phis[1];
    out->phi_points[2] = phis[2];
    out->mass = msum;
    return FMM_OK;
}
