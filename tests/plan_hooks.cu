// Handles for the tests on what no public call reaches: a device of another size, calls
// from two host threads without a pause, eigenvectors without parity.
#include "kx_internal.h"

#include <cmath>
#include <thread>
#include <vector>

// The number of SMs the plan's launches count on; returns the number before.
extern "C" int hook_num_sms(kx_plan *p, int n) {
    const int old = p->num_sms;
    p->num_sms = n;
    return old;
}

// `calls` solves x = f(L) b (one vector) on each of two plans at once, each in a thread and on a
// stream of its own; returns the first error code (0: none).
extern "C" int hook_two_threads(kx_plan *p0, const double *b0, double *x0, kx_plan *p1, const double *b1, double *x1,
                                int calls) {
    int rc[2] = {0, 0};
    auto loop = [&](int i, kx_plan *p, const double *b, double *x) {
        cudaStream_t s;
        if (cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) != cudaSuccess) {
            rc[i] = KX_ERR_CUDA;
            return;
        }
        for (int c = 0; c < calls && !rc[i]; ++c) rc[i] = kx_apply_fL(p, 1, b, x, s);
        if (cudaStreamSynchronize(s) != cudaSuccess && !rc[i]) rc[i] = KX_ERR_CUDA;
        cudaStreamDestroy(s);
    };
    std::thread t(loop, 0, p0, b0, x0);
    loop(1, p1, b1, x1);
    t.join();
    return rc[0] ? rc[0] : rc[1];
}

// Mixes eigenvectors k and k + 1 of an axis by `angle` and makes the float64 tables again.
extern "C" int hook_mix_eigenvectors(kx_plan *p, int axis, int k, double angle) {
    const int n = p->n[axis];
    std::vector<double> V((size_t)n * n);
    if (cudaMemcpy(V.data(), p->d_V[axis], sizeof(double) * V.size(), cudaMemcpyDeviceToHost) != cudaSuccess) return -1;
    const double c = std::cos(angle), s = std::sin(angle);
    for (int x = 0; x < n; ++x) {
        double &a = V[(size_t)x * n + k], &b = V[(size_t)x * n + k + 1];
        const double t = c * a + s * b;
        b = c * b - s * a;
        a = t;
    }
    if (cudaMemcpy(p->d_V[axis], V.data(), sizeof(double) * V.size(), cudaMemcpyHostToDevice) != cudaSuccess) return -1;
    cudaFree(p->d_p64_f);
    p->d_p64_f = nullptr;
    return kx::fp64_setup(p);
}
