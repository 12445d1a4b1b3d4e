// Host harness of test_explicit_step_fault.py: the library's host object linked
// against fakes of the CUDA runtime calls and of the kernels of one explicit
// step, in host memory.  Every fake kernel adds one to what it updates; call
// `fail_call` of them returns an error instead.  Prints, for the given number of
// steps and failing call: status, state.step, state.t, and the range of the
// three arrays.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../include/qsmg.h"
#include "../paper_1904_03808_gb300/csrc/qsmg_impl.h"

extern "C" {
void __cudaInitModule(void **) {}
void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
cudaError_t cudaMalloc(void **p, size_t n) { return (*p = malloc(n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMallocHost(void **p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void *p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void *d, const void *s, size_t n, cudaMemcpyKind, cudaStream_t) { memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void *d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t *s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char *cudaGetErrorString(cudaError_t) { return "fake"; }
}

namespace qsmg {
int calls = 0, fail_call = -1;
cudaError_t kernel(const double *in, double *out, size_t n) {
    if (calls++ == fail_call) return cudaErrorLaunchOutOfResources;
    for (size_t i = 0; i < n; i++) out[i] = in[i] + 1.0;
    return cudaSuccess;
}
size_t cells(const StepParams &p) { return (size_t)p.nx * p.ny * p.nz; }
cudaError_t explicit_stress(const StepParams &p, const double *, const double *sig, const double *,
                            double *out, double *, double *, cudaStream_t) {
    return kernel(sig, out, 6 * cells(p));
}
cudaError_t chi_update(const StepParams &p, const double *, const double *chi, const double *,
                       const double *, double *out, cudaStream_t) {
    return kernel(chi, out, cells(p));
}
cudaError_t explicit_velocity(const StepParams &p, double, double, const double *v, const double *,
                              double *out, cudaStream_t) {
    return kernel(v, out, 3 * (size_t)p.nx * p.ny * (p.nz + 1));
}
cudaError_t wall_fill(const WallParams &, double *, cudaStream_t) {
    return calls++ == fail_call ? cudaErrorLaunchOutOfResources : cudaSuccess;
}
cudaError_t smoother_init() { return cudaSuccess; }
cudaError_t small_init() { return cudaSuccess; }
cudaError_t strip_init() { return cudaSuccess; }
long norm_blocks(const Dims &) { return 1; }
template <typename T>
bool small_plan(const Dims *, const Coarse<T> *, int, int, const double *, int, int, long,
                SmallPlan<T> &) {
    return false;
}
template bool small_plan<float>(const Dims *, const Coarse<float> *, int, int, const double *, int,
                                int, long, SmallPlan<float> &);
template bool small_plan<double>(const Dims *, const Coarse<double> *, int, int, const double *,
                                 int, int, long, SmallPlan<double> &);
}  // namespace qsmg

int main(int argc, char **argv) {
    const int nsteps = atoi(argv[1]);
    const int n = 8;
    mg_grid g{n, n, n, 1e-3};
    mg_moduli m{122e9, 37.4e9};
    mg_bc bc{};
    stz_params z{};
    mg_opts o{};
    mg_ctx *ctx = nullptr;
    if (mg_setup(&g, &m, &bc, &z, &o, nullptr, &ctx) != MG_OK) return 2;
    std::vector<double> a[3] = {std::vector<double>(3 * n * n * (n + 1), 0.0),
                                std::vector<double>(6 * n * n * n, 0.0),
                                std::vector<double>(n * n * n, 0.0)};
    qs_state s{a[0].data(), a[1].data(), a[2].data(), 0.0, 0};
    qsmg::fail_call = argc > 2 ? atoi(argv[2]) : -1;
    const int st = qs_explicit_step(ctx, &s, 1.0, 1.0, 0.0, nsteps);
    printf("%d %ld %g", st, s.step, s.t);
    for (auto &x : a) {
        double lo = x[0], hi = x[0];
        for (double v : x) {
            lo = v < lo ? v : lo;
            hi = v > hi ? v : hi;
        }
        printf(" %g %g", lo, hi);
    }
    printf("\n");
    mg_free(ctx);
    return 0;
}
