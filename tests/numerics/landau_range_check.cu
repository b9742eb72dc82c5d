// The FP64 frame of the fused step (landau_fast: solved in FP32 and corrected
// with FP64 residuals) and the FP64 Newton solve (landau_solve), both against a
// long-double Newton solve of the same moments on the host, at reference
// energies 10^argv[1] to 10^argv[2], speeds up to argv[3], for the spherical
// node (argv[4] = 0: at rest S + eps I = 4/3 eps) and the ring (1: 3/2 eps).
// The error of a state is the largest of its relative errors in eps, gamma and
// v (relative to |v|).  Prints one JSON list of [exponent, fast max, fast mean,
// solve max, solve mean].  Test infrastructure only.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2101_06187_gb300/csrc/rlbm_device.cuh"

using namespace rlbk;

struct Moments {
    double eps0, dE, Mx, My, Sxx, Sxy, Syy;
};
struct Out {
    double f[2][4];  // fast, solve: eps, vx, vy, gamma
};

Moments sample(int i, int n, double vmax, double eps0, double rest) {
    const double t = (double)i / n;
    const double eps = eps0 * (0.7 + 0.6 * fmod(t * 7.31, 1.0));
    const double sp = vmax * (0.05 + 0.95 * fmod(t * 3.17 + 0.13, 1.0)), th = 6.283185307179586 * fmod(t * 11.7, 1.0);
    const double vx = sp * cos(th), vy = sp * sin(th), w = rest * eps / (1.0 - vx * vx - vy * vy);
    const double P = (rest - 1.0) * eps, ne = 1e-3 * eps0 * sin(17.0 * t);
    return Moments{eps0, w - P - eps0, w * vx, w * vy, w * vx * vx + P - (rest - 1.0) * eps0 + ne, w * vx * vy + 0.5 * ne,
                   w * vy * vy + P - (rest - 1.0) * eps0 - ne};
}

__global__ void k_frames(int n, const Moments *in, Out *out, double rest) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Moments m = in[i];
    const Frame<double> f[2] = {landau_fast<double>(m.eps0, m.dE, m.Mx, m.My, m.Sxx, m.Sxy, m.Syy, rest),
                                landau_solve<double>(m.eps0, m.dE, m.Mx, m.My, m.Sxx, m.Sxy, m.Syy, rest)};
    for (int k = 0; k < 2; ++k) {
        out[i].f[k][0] = f[k].eps;
        out[i].f[k][1] = f[k].vx;
        out[i].f[k][2] = f[k].vy;
        out[i].f[k][3] = f[k].gamma;
    }
}

int main(int argc, char **argv) {
    if (argc != 5) return 2;
    const int lo = std::atoi(argv[1]), hi = std::atoi(argv[2]), per = 512, n = (hi - lo + 1) * per;
    const double rest = std::atoi(argv[4]) ? 1.5 : 4.0 / 3.0;
    std::vector<Moments> h(n);
    for (int i = 0; i < n; ++i)
        h[i] = sample(i % per, per, std::atof(argv[3]), std::pow(10.0, lo + i / per), rest);
    Moments *d = nullptr;
    Out *dout = nullptr;
    if (cudaMalloc(&d, sizeof(Moments) * n) != cudaSuccess || cudaMalloc(&dout, sizeof(Out) * n) != cudaSuccess) return 1;
    if (cudaMemcpy(d, h.data(), sizeof(Moments) * n, cudaMemcpyHostToDevice) != cudaSuccess) return 1;
    k_frames<<<(n + 127) / 128, 128>>>(n, d, dout, rest);
    std::vector<Out> out(n);
    if (cudaMemcpy(out.data(), dout, sizeof(Out) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    std::printf("[");
    for (int e = 0; e <= hi - lo; ++e) {
        double worst[2] = {0, 0}, mean[2] = {0, 0};
        for (int i = e * per; i < (e + 1) * per; ++i) {
            typedef long double L;
            const Moments m = h[i];
            const L a0 = (L)rest * m.eps0 + m.dE, Mx = m.Mx, My = m.My;
            L delta = 0, vx = 0, vy = 0;
            for (int it = 0; it < 16; ++it) {
                const L xx = a0 - delta + m.Sxx, yy = a0 - delta + m.Syy, det = xx * yy - (L)m.Sxy * m.Sxy;
                vx = (yy * Mx - m.Sxy * My) / det;
                vy = (xx * My - m.Sxy * Mx) / det;
                delta -= (delta - (Mx * vx + My * vy)) / (1 - vx * vx - vy * vy);
            }
            const L want[4] = {m.eps0 + (m.dE - delta), vx, vy, 1 / sqrtl(1 - vx * vx - vy * vy)};
            const L vn = sqrtl(vx * vx + vy * vy);
            for (int k = 0; k < 2; ++k) {
                L err = 0;
                for (int j = 0; j < 4; ++j) {
                    const L x = fabsl(out[i].f[k][j] - want[j]) / (j == 1 || j == 2 ? vn : want[j]);
                    if (!(x <= err)) err = x;  // NaN sticks
                }
                if (!((double)err <= worst[k])) worst[k] = (double)err;
                mean[k] += (double)err / per;
            }
        }
        auto num = [](double x) { return std::isfinite(x) ? x : 1e300; };  // JSON has no NaN
        std::printf("%s[%d, %.4e, %.4e, %.4e, %.4e]", e ? ", " : "", lo + e, num(worst[0]), num(mean[0]), num(worst[1]),
                    num(mean[1]));
    }
    std::printf("]\n");
    return 0;
}
