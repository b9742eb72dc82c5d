// Errors of the fused step's Landau frame (landau_fast in rlbm_device.cuh) and
// of the Newton solve it stands in for (landau_solve), both against a
// long-double Newton solve of the same moments on the host, for fluid states
// with |v| up to argv[1], reference energy argv[2] and velocities scaled by
// argv[3] (tiny momenta): FP64 (solved in FP32 and corrected with FP64
// residuals, or by the FP64 Newton solve where FP32 cannot carry it) and
// packed FP32 lanes (the early exit and the Newton continuation; the other
// lane holds another state, so both meet in one pair).  The error of a state
// is the largest of its relative errors in eps, gamma and v (relative to |v|).
// Prints one JSON line.  Test infrastructure only.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2101_06187_gb300/csrc/packed.cuh"

using namespace rlbk;

struct Moments {
    double eps0, dE, Mx, My, Sxx, Sxy, Syy;
};
struct Out {
    double f[4][4];  // solve FP64, fast FP64, solve FP32, fast FP32: eps, vx, vy, gamma
};

__host__ __device__ Moments sample(int i, int n, double vmax, double eps0, double tiny) {
    const double t = (double)i / n;
    const double eps = eps0 * (0.7 + 0.6 * fmod(t * 7.31, 1.0));
    const double sp = tiny * vmax * fmod(t * 3.17 + 0.13, 1.0), th = 6.283185307179586 * fmod(t * 11.7, 1.0);
    const double vx = sp * cos(th), vy = sp * sin(th), g2 = 1.0 / (1.0 - vx * vx - vy * vy);
    const double w = 4.0 / 3.0 * eps * g2, ne = 1e-3 * eps0 * sin(17.0 * t);
    // rounded to FP32 where that holds it, so one reference serves both precisions
    auto r = [&](double x) { return fabs(x) > 1e-30 && fabs(x) < 1e30 ? (double)(float)x : x; };
    return Moments{r(eps0), r(w - eps / 3.0 - eps0), r(w * vx), r(w * vy), r(w * vx * vx + (eps - eps0) / 3.0 + ne),
                   r(w * vx * vy + 0.5 * ne), r(w * vy * vy + (eps - eps0) / 3.0 - ne)};
}

template <typename F>
__device__ void put(double (&o)[4], const F &f, double (*get)(const F &, int)) {
    for (int k = 0; k < 4; ++k) o[k] = get(f, k);
}
__device__ double get64(const Frame<double> &f, int k) { return k == 0 ? f.eps : k == 1 ? f.vx : k == 2 ? f.vy : f.gamma; }
__device__ double get32(const Frame<pf2> &f, int k) {
    return k == 0 ? f.eps.v.x : k == 1 ? f.vx.v.x : k == 2 ? f.vy.v.x : f.gamma.v.x;
}

__global__ void k_frames(int n, const Moments *in, Out *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Moments m = in[i], o = in[(i + n / 2) % n];
    put(out[i].f[0], landau_solve<double>(m.eps0, m.dE, m.Mx, m.My, m.Sxx, m.Sxy, m.Syy), get64);
    put(out[i].f[1], landau_fast<double>(m.eps0, m.dE, m.Mx, m.My, m.Sxx, m.Sxy, m.Syy), get64);
    auto two = [](double a, double b) { return pf2((float)a, (float)b); };
    const pf2 a[7] = {two(m.eps0, o.eps0), two(m.dE, o.dE),   two(m.Mx, o.Mx),  two(m.My, o.My),
                      two(m.Sxx, o.Sxx),   two(m.Sxy, o.Sxy), two(m.Syy, o.Syy)};
    put(out[i].f[2], landau_solve<pf2>(a[0], a[1], a[2], a[3], a[4], a[5], a[6]), get32);
    put(out[i].f[3], landau_fast<pf2>(a[0], a[1], a[2], a[3], a[4], a[5], a[6]), get32);
}

// widen() against the conversion instruction: every 2^9 + 1st float, zeros, subnormals, infinities and NaN among them.
__global__ void k_widen(int *bad) {
    for (unsigned long long u = threadIdx.x + (unsigned long long)blockIdx.x * blockDim.x; u < (1ull << 32) / 513;
         u += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned b = (unsigned)(u * 513);
        const float x = __uint_as_float(b ^ (b >> 3 & 1u ? 0u : 0x80000000u));
        if (__double_as_longlong(widen(x)) != __double_as_longlong((double)x) && x == x) atomicAdd(bad, 1);
    }
    if (blockIdx.x == 0 && threadIdx.x < 10) {
        const unsigned edge[5] = {0u, 1u, 0x007fffffu, 0x00800000u, 0x7f800000u};
        const float x = __uint_as_float(edge[threadIdx.x / 2] | (threadIdx.x & 1 ? 0x80000000u : 0u));
        if (__double_as_longlong(widen(x)) != __double_as_longlong((double)x)) atomicAdd(bad, 1);
    }
}

int main(int argc, char **argv) {
    if (argc != 4) return 2;
    const int n = 1 << 15;
    std::vector<Moments> h(n);
    for (int i = 0; i < n; ++i) h[i] = sample(i, n, std::atof(argv[1]), std::atof(argv[2]), std::atof(argv[3]));
    Moments *d = nullptr;
    Out *dout = nullptr;
    if (cudaMalloc(&d, sizeof(Moments) * n) != cudaSuccess || cudaMalloc(&dout, sizeof(Out) * n) != cudaSuccess) return 1;
    cudaMemcpy(d, h.data(), sizeof(Moments) * n, cudaMemcpyHostToDevice);
    k_frames<<<n / 128, 128>>>(n, d, dout);
    std::vector<Out> out(n);
    if (cudaMemcpy(out.data(), dout, sizeof(Out) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    double worst[4] = {0, 0, 0, 0}, mean[4] = {0, 0, 0, 0};
    for (int i = 0; i < n; ++i) {
        typedef long double L;
        const Moments m = h[i];
        const L a0 = (L)4 / 3 * m.eps0 + m.dE, Mx = m.Mx, My = m.My;
        L delta = 0, vx = 0, vy = 0;
        for (int it = 0; it < 60; ++it) {
            const L xx = a0 - delta + m.Sxx, yy = a0 - delta + m.Syy, det = xx * yy - (L)m.Sxy * m.Sxy;
            vx = (yy * Mx - m.Sxy * My) / det;
            vy = (xx * My - m.Sxy * Mx) / det;
            delta -= (delta - (Mx * vx + My * vy)) / (1 - vx * vx - vy * vy);
        }
        const L want[4] = {m.eps0 + (m.dE - delta), vx, vy, 1 / sqrtl(1 - vx * vx - vy * vy)};
        const L vn = fmaxl(sqrtl(vx * vx + vy * vy), 1e-300L);
        for (int k = 0; k < 4; ++k) {
            L e = 0;
            for (int j = 0; j < 4; ++j) {
                const L x = fabsl(out[i].f[k][j] - want[j]) / (j == 1 || j == 2 ? vn : want[j]);
                if (!(x <= e)) e = x;  // NaN sticks
            }
            if (!((double)e <= worst[k])) worst[k] = (double)e;
            mean[k] += (double)e / n;
        }
    }
    const char *name[4] = {"solve64", "fast64", "solve32", "fast32"};
    int *dbad = nullptr, bad = 1;
    if (cudaMalloc(&dbad, sizeof(int)) != cudaSuccess || cudaMemset(dbad, 0, sizeof(int)) != cudaSuccess) return 1;
    k_widen<<<608, 256>>>(dbad);
    if (cudaMemcpy(&bad, dbad, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    std::printf("{\"widen_bad\": %d, ", bad);
    for (int k = 0; k < 4; ++k) {
        auto num = [](double x) { return std::isfinite(x) ? x : 1e300; };  // JSON has no NaN
        std::printf("\"%s_max\": %.4e, \"%s_mean\": %.4e%s", name[k], num(worst[k]), name[k], num(mean[k]),
                    k < 3 ? ", " : "}\n");
    }
    return 0;
}
