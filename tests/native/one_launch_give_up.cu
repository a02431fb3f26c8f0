// One handle whose one-launch substitutions give up on their waits (a poll limit of 1) and then, with the
// normal limit, run on the same barrier counters: the give-up is a status that says what it is, the
// counters are back at zero, and the next application on the handle equals the one before the give-up.
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "hz_internal.cuh"
#include "hz_ctx.cuh"
#include "hz_solve.cuh"

#define CHECK(cond)                                                      \
    do {                                                                 \
        if (!(cond)) {                                                   \
            std::printf("%s:%d: %s\n", __FILE__, __LINE__, #cond);       \
            std::exit(1);                                                \
        }                                                                \
    } while (0)

int main() {
    const int n = 24, L = 3, R = 3;
    std::vector<double> m((size_t)n * n * n);
    unsigned seed = 1;
    for (double& v : m) {
        seed = seed * 1664525u + 1013904223u;
        const double c = 1.5 + (seed >> 8) / (double)(1 << 24);
        v = 1.0 / (c * c);
    }
    hz_grid grid{n, n, n, 1.0};
    hz_pml pml{4, 10.0, -1};
    setenv("HZ_FACTOR_TC_MIN", "0", 1);   // no bounded waits in the factorization
    hz_handle* h = nullptr;
    CHECK(hz_create_ex(&grid, m.data(), nullptr, 0.9, &pml, L, HZ_PREC_MIXED, nullptr, &h) == HZ_OK);
    CHECK(hz_factor(h) == HZ_OK);
    const long long ntr = (long long)R * 2 * (L - 1) * 2 * n * n;
    std::vector<std::complex<double>> x(ntr), y0(ntr), y1(ntr);
    for (auto& v : x) {
        seed = seed * 1664525u + 1013904223u;
        v = {(seed >> 8) / (double)(1 << 24) - 0.5, (seed & 255) / 256.0 - 0.5};
    }
    double *dx = nullptr, *dy = nullptr;
    CHECK(cudaMalloc(&dx, ntr * 16) == cudaSuccess && cudaMalloc(&dy, ntr * 16) == cudaSuccess);
    CHECK(cudaMemcpy(dx, x.data(), ntr * 16, cudaMemcpyHostToDevice) == cudaSuccess);
    auto words = [&]() {
        std::vector<int> w(4);
        CHECK(cudaMemcpy(w.data(), h->ctx.d_flag, 16, cudaMemcpyDeviceToHost) == cudaSuccess);
        return w;
    };
    auto apply = [&](long long polls) {
        CHECK(cudaDeviceSynchronize() == cudaSuccess);
        hz::free_batches(h->ctx);   // batches keep the limit they were made with
        h->ctx.tc_wait_polls = polls;
        return hz_apply_precond(h, dx, R, dy);
    };
    CHECK(apply(1LL << 26) == HZ_OK);
    CHECK(hz::use_one_launch(h->ctx, 4, 0));
    CHECK(cudaMemcpy(y0.data(), dy, ntr * 16, cudaMemcpyDeviceToHost) == cudaSuccess);
    for (int rep = 0; rep < 3; ++rep) {
        CHECK(apply(1) == HZ_ERR_TIMEOUT);
        CHECK(std::strstr(hz_last_error(h), "wait") && !std::strstr(hz_last_error(h), "MMA"));
        const std::vector<int> w = words();
        CHECK(w[1] == 0 && w[2] == 0 && w[3] == 0);   // reported and cleared; both counters at zero
        CHECK(apply(1LL << 26) == HZ_OK);
        CHECK(cudaMemcpy(y1.data(), dy, ntr * 16, cudaMemcpyDeviceToHost) == cudaSuccess);
        double d = 0, s = 0;
        for (long long i = 0; i < ntr; ++i) { d += std::norm(y1[i] - y0[i]); s += std::norm(y0[i]); }
        CHECK(s > 0 && std::sqrt(d / s) < 5e-6);      // FP32 rounding in another order of the additions
    }
    // the whole solve reports it too
    std::vector<std::complex<double>> f((size_t)n * n * n);
    f[(size_t)(n / 2) * n * n + n / 2 * n + n / 2] = 1.0;
    double *df = nullptr, *du = nullptr;
    CHECK(cudaMalloc(&df, f.size() * 16) == cudaSuccess && cudaMalloc(&du, f.size() * 16) == cudaSuccess);
    CHECK(cudaMemcpy(df, f.data(), f.size() * 16, cudaMemcpyHostToDevice) == cudaSuccess);
    hz::free_batches(h->ctx);
    h->ctx.tc_wait_polls = 1;
    hz_solve_opts o;
    hz_default_opts(HZ_PREC_MIXED, &o);
    o.max_iter = 2;
    o.max_refine = 0;
    CHECK(hz_solve(h, df, 1, du, &o, nullptr) == HZ_ERR_TIMEOUT);
    CHECK(std::strstr(hz_last_error(h), "wait") && !std::strstr(hz_last_error(h), "MMA"));
    CHECK(hz_destroy(h) == HZ_OK);
    CHECK(cudaDeviceSynchronize() == cudaSuccess);
    std::printf("ok\n");
    return 0;
}
