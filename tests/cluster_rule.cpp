// The coarsest-grid solver takes the largest clusters of which the device holds all instances at once.  The
// runtime calls defined here take the place of libcudart's for the solver library: a device that holds 7
// clusters of 16 thread blocks, 15 of 8, 36 of 4 and 76 of 2; launches are recorded, not run.
#include <cstdio>

#include "ohm_internal.h"

static unsigned g_cluster = 0, g_grid = 0;
static unsigned cluster_of(const cudaLaunchConfig_t *c) {
    for (unsigned i = 0; i < c->numAttrs; i++)
        if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
    return 1;
}
extern "C" {
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *c, const void *, void **) {
    g_cluster = cluster_of(c);
    g_grid = c->gridDim.x;
    return cudaSuccess;
}
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int *n, const void *, const cudaLaunchConfig_t *c) {
    const unsigned cs = cluster_of(c);
    *n = cs == 16 ? 7 : (cs == 8 ? 15 : (cs == 4 ? 36 : 76));
    return cudaSuccess;
}
}

using namespace ohm;

template <typename T>
static int check(int ninst, int edge, unsigned want) {
    SmallDev<T> sm = {};
    sm.ninst = ninst;
    sm.omega = 1.0;
    for (int e = edge; e >= 2; e /= 2, sm.n++) {
        sm.dims[sm.n][0] = sm.dims[sm.n][1] = sm.dims[sm.n][2] = e;
        sm.h[sm.n] = 1.0;
    }
    const cudaError_t e = launch_tail<T>(sm, 1.0, 1, 1, 1, nullptr);
    if (e == cudaSuccess && g_cluster == want && g_grid == want * ninst) return 0;
    printf("float%d, %d instances of %d^3: clusters of %u (grid %u, error %d), want %u\n", (int)sizeof(T) * 8, ninst, edge, g_cluster,
           g_grid, e, want);
    return 1;
}

int main() {
    int bad = 0;
    const struct { int ninst; unsigned f32, f64; } rule[] = {{1, 8, 16},  {7, 8, 16},  {8, 8, 8},   {15, 8, 8},  {16, 4, 4},
                                                             {36, 4, 4}, {37, 2, 2}, {76, 2, 2}, {77, 1, 1}, {500, 1, 1}};
    for (auto &r : rule) {
        bad += check<float>(r.ninst, 16, r.f32);
        bad += check<double>(r.ninst, 16, r.f64);
    }
    bad += check<float>(1, 8, 1);   // a first grid that is not divided: one thread block
    bad += check<double>(1, 4, 1);
    if (bad == 0) printf("ok\n");
    return bad != 0;
}
