// spmv_stokes on the host, one warp at a time with a thread per lane: the
// kernel's text (kernel.inc) with the few CUDA names it uses.  A shuffle with
// the full mask wants every lane that has not returned, so all lanes that
// shuffle at all have to shuffle equally often.  Prints the largest error
// against a sum in double, relative to the sum of magnitudes, and exits with 1
// if the lanes of a warp disagree.
#include <barrier>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <thread>
#include <vector>

#define __global__
#define __launch_bounds__(n)
#define __restrict__
struct Dim { int x = 0; };
static Dim blockIdx, blockDim;
static thread_local Dim threadIdx;
static thread_local int shuffles;
static float slot[32];
static std::barrier<>* bar;
template <typename T> T __ldg(const T* p) { return *p; }
static void pdl_wait() {}
static void pdl_release() {}
static float __shfl_down_sync(unsigned, float v, int o, int width) {
    const int lane = threadIdx.x & 31;
    ++shuffles;
    slot[lane] = v;
    bar->arrive_and_wait();
    const float r = lane % width + o < width ? slot[lane + o] : v;
    bar->arrive_and_wait();
    return r;
}
enum SpmvMode { SPMV_SET = 0, SPMV_ADD = 1, SPMV_RESID = 2 };
#include "kernel.inc"

template <int LANES, int D>
static bool check(int nvf, int nq, int per_row, double* worst) {
    std::mt19937 rng(nvf * 131 + nq);
    std::uniform_real_distribution<float> val(-1.f, 1.f);
    const int n = D * nvf + nq;
    std::vector<int> rp(n + 1, 0), ci;
    std::vector<float> av, x(n), b(n), y(n, 0.f);
    for (int i = 0; i < n; ++i) { x[i] = val(rng); b[i] = val(rng); }
    std::vector<std::vector<int>> nv(nvf + nq), np(nvf);
    std::vector<std::vector<float>> a(nvf);
    for (int g = 0; g < nvf + nq; ++g)
        for (int k = 0; k < 1 + (int)(rng() % per_row); ++k) nv[g].push_back(rng() % nvf);
    for (int g = 0; g < nvf; ++g) {
        for (int k = 0; k < (int)(rng() % 4); ++k) np[g].push_back(rng() % nq);
        for (size_t k = 0; k < nv[g].size(); ++k) a[g].push_back(val(rng));
    }
    for (int i = 0; i < n; ++i) {
        const int c = i < D * nvf ? i / nvf : 0, g = i < D * nvf ? i % nvf : nvf + i - D * nvf;
        if (g < nvf) {
            for (size_t k = 0; k < nv[g].size(); ++k) { ci.push_back(c * nvf + nv[g][k]); av.push_back(a[g][k]); }
            for (int q : np[g]) { ci.push_back(D * nvf + q); av.push_back(val(rng)); }
        } else {
            for (int cc = 0; cc < D; ++cc)
                for (int j : nv[g]) { ci.push_back(cc * nvf + j); av.push_back(val(rng)); }
        }
        rp[i + 1] = (int)ci.size();
    }
    blockDim.x = 256;
    bool same = true;
    const int threads = (nvf + nq) * LANES;
    for (int w = 0; w < (threads + 255) / 256 * 8; ++w) {
        blockIdx.x = w / 8;
        std::barrier<> warp(32);
        bar = &warp;
        int count[32];
        std::vector<std::thread> lanes;
        for (int l = 0; l < 32; ++l)
            lanes.emplace_back([&, l] {
                threadIdx.x = (w % 8) * 32 + l;
                shuffles = 0;
                spmv_stokes<LANES, SPMV_RESID, D>(nvf, nq, rp.data(), ci.data(), av.data(), x.data(), y.data(), b.data());
                count[l] = shuffles;
                warp.arrive_and_drop();
            });
        for (auto& t : lanes) t.join();
        for (int l = 0; l < 32; ++l) same &= count[l] == 0 || count[l] == count[0];
    }
    for (int i = 0; i < n; ++i) {
        double s = b[i], m = std::fabs(b[i]);
        for (int k = rp[i]; k < rp[i + 1]; ++k) { s -= (double)av[k] * x[ci[k]]; m += std::fabs((double)av[k] * x[ci[k]]); }
        *worst = std::fmax(*worst, std::fabs(y[i] - s) / m);
    }
    return same;
}

int main() {
    double worst = 0;
    bool same = true;
    // warps of velocity nodes alone, of both kinds, and of live and idle lanes
    for (int nvf : {3, 8, 13, 30})
        for (int nq : {1, 6, 11}) {
            same &= check<8, 2>(nvf, nq, 70, &worst) & check<8, 3>(nvf, nq, 70, &worst);
            same &= check<4, 2>(nvf, nq, 40, &worst) & check<4, 3>(nvf, nq, 40, &worst);
            same &= check<16, 2>(nvf, nq, 70, &worst) & check<32, 3>(nvf, nq, 70, &worst);
        }
    std::printf("%.3e\n", worst);
    return same ? 0 : 1;
}
