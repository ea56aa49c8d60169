// Every kernel launcher under a CUDA runtime whose launches fail: the error is returned, once, and none is
// left behind for the process's next cudaGetLastError (which would report it from a call that succeeded).
// The runtime calls defined here take the place of libcudart's for the solver library too.
#include <cstdio>

#include "ohm_internal.h"

static cudaError_t g_last = cudaSuccess;
static bool g_fail = false;
static int g_launches = 0;
static cudaError_t launch() {
    g_launches++;
    if (g_fail) g_last = cudaErrorLaunchOutOfResources;
    return g_fail ? cudaErrorLaunchOutOfResources : cudaSuccess;
}
extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *, const void *, void **) { return launch(); }
cudaError_t __cudaLaunchKernel(void *, dim3, dim3, void **, size_t, cudaStream_t) { return launch(); }
cudaError_t __cudaGetKernel(void **k, const void *f) {
    *k = const_cast<void *>(f);
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
    const cudaError_t e = g_last;
    g_last = cudaSuccess;
    return e;
}
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *) {
    *n = 1;
    return cudaSuccess;
}
}

using namespace ohm;

static int bad = 0;
#define TEST(call)                                                                                          \
    do {                                                                                                    \
        g_fail = true;                                                                                      \
        g_launches = 0;                                                                                     \
        const cudaError_t e1 = (call), left = g_last;                                                       \
        g_last = cudaSuccess;                                                                               \
        g_fail = false;                                                                                     \
        const cudaError_t e2 = (call);                                                                      \
        if (e1 != cudaErrorLaunchOutOfResources || left != cudaSuccess || e2 != cudaSuccess || !g_launches) { \
            printf("%s: returned %d, left %d, then %d (%d launches)\n", #call, e1, left, e2, g_launches);   \
            bad++;                                                                                          \
        }                                                                                                   \
    } while (0)

template <typename T>
static SmallDev<T> small() {
    SmallDev<T> sm = {};
    sm.n = 2;
    sm.ninst = 1;
    sm.omega = 1.0;
    for (int s = 0; s < 2; s++) {
        sm.dims[s][0] = sm.dims[s][1] = sm.dims[s][2] = s ? 2 : 4;
        sm.h[s] = 1.0;
    }
    return sm;
}

template <typename T>
static void both(const GridDev &g) {  // kernels of either precision
    T *p = nullptr;
    const int ld[3] = {4, 4, 4};
    TEST((launch_smooth<T>(g, p, p, p, p, p, p, p, 1.0, 0, nullptr)));
    TEST((launch_smooth_zero(g, p, p, p, p, p, 1.0, nullptr)));
    TEST((launch_resid_restrict<T>(g, p, p, p, p, p, 1.0, nullptr, nullptr, p, ld, nullptr)));
    TEST((launch_prolong_add<T>(g, nullptr, nullptr, p, ld, p, nullptr, nullptr)));
    TEST((launch_restrict<T>(g, p, 1, p, nullptr, nullptr, nullptr)));
    TEST((launch_ghost_fill<T, T>(g, g, p, 3, p, nullptr, nullptr)));
    TEST((launch_sync_down<T>(g, p, p, nullptr)));
    TEST((launch_axpy_leaf<T>(g, p, p, nullptr, nullptr)));
    TEST((launch_update<T>(g, nullptr, p, nullptr, nullptr)));
    TEST((launch_invdiag<T>(g, p, p, 1.0, p, nullptr)));
    const SmallDev<T> sm = small<T>();
    TEST((launch_tail<T>(sm, 1.0, 1, 1, 1, nullptr)));
    TEST((launch_lex_sweeps<T>(sm, 0, 1.0, 1, nullptr)));
    TEST((launch_lex_resid_restrict<T>(sm, 0, 1.0, nullptr)));
    TEST((launch_lex_prolong<T>(sm, 0, nullptr)));
    TEST((launch_small_eta<T>(sm, nullptr)));
    TEST((launch_small_inv<T>(sm, 1.0, nullptr)));
}

int main() {
    double *d = nullptr;
    float *f = nullptr;
    dfloat *df = nullptr;
    for (int nblk : {2, 512, 4096}) {  // both launch kinds and every slab height
        GridDev g;
        g.nblk = nblk;
        g.h = 1.0;
        g.nslot = 1;
        both<double>(g);
        both<float>(g);
        TEST((launch_composite<double>(g, d, d, d, d, d, -1.0, 1.0, 1.0, d, d, d, nullptr, nullptr, nullptr)));
        TEST((launch_composite<double>(g, d, nullptr, d, d, d, 1.0, 1.0, 0.0, d, d, d, nullptr, nullptr, nullptr)));
        double one;  // (norm partials: any non-null pointer)
        TEST((launch_composite<float>(g, d, &one, d, d, d, -1.0, 1.0, 1.0, f, f, d, nullptr, &one, nullptr)));
        TEST((launch_composite<float>(g, d, nullptr, d, d, d, 1.0, 1.0, 0.0, f, f, d, nullptr, &one, nullptr, &one, 1.0)));
        TEST((launch_composite(g, f, f, f, f, f, -1.0, 1.0, 1.0, f, f, d, nullptr, d, 1.0, nullptr)));
        TEST((launch_composite_df(g, d, df, d, d, d, -1.0, 1.0, 1.0, f, f, d, nullptr, d, 1.0, nullptr, df, 0.0)));
        TEST((launch_composite_df(g, d, d, d, d, d, -1.0, 1.0, 1.0, f, f, d, nullptr, d, 1.0, nullptr)));
        float x;
        TEST((launch_smooth_rb(g, f, f, f, f, 1.0, nullptr)));
        TEST((launch_smooth_rb(g, &x, f, f, f, 1.0, nullptr)));
        TEST((launch_smooth_rb2(g, f, f, f, f, 1.0, nullptr)));
        TEST((launch_pair_op(g, f, f, f, 1.0, true, f, nullptr, nullptr)));
        TEST((launch_prolong_add8<float>(g, f, f, nullptr)));
    }
    if (bad == 0) printf("ok\n");
    return bad != 0;
}
