// The host code of the library against a fake of the CUDA runtime and of its
// launches, which keeps count of what each stream has been given and of what it
// waits for.  For every launch of fmm_m2l and fmm_step in turn, that launch
// fails; whatever was enqueued by then, on either stream, must be ordered
// before what the caller enqueues on the stream next.  With an argument: prints
// the monopole weights of the FP64 kernels at that opening angle.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>

#include "fmm_internal.h"

namespace {

int g_next = 0;                        // operations enqueued so far
int g_launch = 0, g_fail_at = -1;      // launches asked for, the one that fails
std::map<const void *, std::set<int>> g_seen;     // stream or event -> operations it stands after

const cudaStream_t kUser = reinterpret_cast<cudaStream_t>(16);

cudaError_t enqueue(cudaStream_t s)
{
    if (g_launch++ == g_fail_at) return cudaErrorLaunchFailure;
    g_seen[s].insert(g_next++);
    return cudaSuccess;
}

}  // namespace

extern "C" {
cudaError_t cudaMalloc(void **p, size_t n) { *p = std::malloc(n ? n : 1); return cudaSuccess; }
cudaError_t cudaFree(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void **p, size_t n) { *p = std::malloc(n); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void *, const void *, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemset(void *, int, size_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int *d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int *v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t *e) { *e = reinterpret_cast<cudaEvent_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float *ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { g_seen[e] = g_seen[s]; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned)
{
    g_seen[s].insert(g_seen[e].begin(), g_seen[e].end());
    return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = reinterpret_cast<cudaStream_t>(std::malloc(1)); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
}

namespace fmm {
cudaError_t launch_p2m(const fmm_tree_s *, const double *, double *, cudaStream_t s, bool) { return enqueue(s); }
cudaError_t launch_m2m_level(const fmm_tree_s *, int, double *, double *, cudaStream_t s) { return enqueue(s); }
int m2m_split(const fmm_tree_s *, int, ListRange &, ListRange &) { return 1; }
cudaError_t launch_pack(const fmm_tree_s *, const double *, const double *, cudaStream_t s, int) { return enqueue(s); }
cudaError_t launch_m2l(const fmm_tree_s *, void *, float *, double *, cudaStream_t s, int *, int) { return enqueue(s); }
cudaError_t launch_l2l_level(const fmm_tree_s *, int, const void *, const float *, const double *, const double *,
                             double *, double *, cudaStream_t s) { return enqueue(s); }
cudaError_t launch_l2l_leaves(const fmm_tree_s *, const void *, const float *, const double *, const double *,
                              double *, double *, cudaStream_t s) { return enqueue(s); }
cudaError_t launch_leaf_finish(const fmm_tree_s *, const void *, const float *, const double *, const double *,
                               double *, double *, const double *, double *, double *, cudaStream_t s) { return enqueue(s); }
cudaError_t launch_downward_dataflow(const fmm_tree_s *, const void *, const float *, const double *, const double *,
                                     double *, double *, const double *, double *, double *, cudaStream_t s) { return enqueue(s); }
cudaError_t launch_forces(const fmm_tree_s *, const double *, const double *, const double *, double *, double *,
                          double *, cudaStream_t s) { return enqueue(s); }
cudaError_t launch_force_sums(const fmm_tree_s *, double *, cudaStream_t s) { return enqueue(s); }
}  // namespace fmm

// a root, its 8 children, and with levels = 3 theirs
static fmm_tree_t build(int levels, double theta = 0.5, int precision = FMM_MIXED)
{
    std::vector<fmm_node_desc> d;
    std::vector<int> first;
    for (int lev = 1; lev <= levels; ++lev) {
        first.push_back(int(d.size()));
        const int side = 1 << (lev - 1);
        for (int i = 0; i < side * side * side; ++i) {
            fmm_node_desc x{};
            x.level = lev;
            x.ix = i % side;
            x.iy = i / side % side;
            x.iz = i / side / side;
            x.parent = lev == 1 ? -1 : first[lev - 2] + x.ix / 2 + side / 2 * (x.iy / 2 + side / 2 * (x.iz / 2));
            for (int k = 0; k < 8; ++k) x.child[k] = -1;
            d.push_back(x);
        }
    }
    for (size_t i = 1; i < d.size(); ++i)
        d[size_t(d[i].parent)].child[(d[i].ix & 1) + 2 * (d[i].iy & 1) + 4 * (d[i].iz & 1)] = int(i);
    fmm_config c{};
    c.theta = theta;
    c.G = 1.0;
    c.box_size = 1.0;
    c.precision = precision;
    c.max_level = 20;
    fmm_tree_t t = nullptr;
    if (fmm_build_tree(d.data(), int64_t(d.size()), &c, &t) != FMM_OK) {
        std::printf("build: %s\n", fmm_last_error());
        std::exit(2);
    }
    return t;
}

int main(int argc, char **argv)
{
    if (argc > 1) {
        // the FP64 monopole weights' table at an opening angle
        fmm_tree_t t = build(2, std::atof(argv[1]), FMM_FP64);
        std::printf("%zu\n", t->orbits.size() / 4);
        for (int32_t v : t->orbits) std::printf("%d\n", v);
        for (double v : t->orbit_coef) std::printf("%a\n", v);
        fmm_destroy_tree(t);
        return 0;
    }
    int bad = 0, tried = 0;
    alignas(16) static double buf[2];
    float f;
    for (int levels = 2; levels <= 3; ++levels) {
        fmm_tree_t t = build(levels);
        for (int dataflow = 0; dataflow < 2; ++dataflow) {
            fmm_tuning tu{};
            tu.dataflow = dataflow;
            fmm_set_tuning(t, &tu);
            for (int step = 0; step < 2; ++step) {
                for (int at = 0;; ++at) {
                    g_seen.clear();
                    g_next = g_launch = 0;
                    g_fail_at = at;
                    const int rc = step ? fmm_step(t, buf, buf, buf, buf, &f, buf, buf, buf, buf, buf, buf, kUser)
                                        : fmm_m2l(t, buf, buf, buf, &f, buf, kUser);
                    const bool ran = g_launch <= at;         // no such launch: the call went through
                    if ((rc == FMM_OK) != ran) { std::printf("rc %d, launch %d\n", rc, at); ++bad; }
                    if (int(g_seen[kUser].size()) != g_next) {
                        std::printf("%s, %d levels, launch %d fails: %d of %d operations joined\n",
                                    step ? "fmm_step" : "fmm_m2l", levels, at, int(g_seen[kUser].size()), g_next);
                        ++bad;
                    }
                    ++tried;
                    if (ran) break;
                }
            }
        }
        fmm_destroy_tree(t);
    }
    std::printf("%d calls, %d faults\n", tried, bad);
    return bad ? 1 : 0;
}
