// The fused step's FP32 frame (landau_fast) on packed lanes: whether a node's
// frame depends on the node in the other lane, and how far the frames of many
// states lean to one side.  States with |v| between argv[1] and argv[2], each
// paired with itself, with its neighbour in the list and with a state at rest,
// in either lane.  Prints one JSON line: frames whose bits differ between the
// pairings, and the mean signed relative error of v along v and the mean of
// (delta - M . v) / delta over the states, against a long-double solve (delta =
// E - eps).  Test infrastructure only.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../paper_2101_06187_gb300/csrc/packed.cuh"

using namespace rlbk;

struct Moments {
    float dE, Mx, My, Sxx, Sxy, Syy;
};
struct Out {
    float f[7];  // ddelta_eps, eps, vx, vy, v2, g2, gamma
};

Moments sample(int i, int n, double lo, double hi) {
    const double t = (double)i / n;
    const double eps = 0.998 + 0.004 * fmod(t * 7.31, 1.0), sp = lo + (hi - lo) * fmod(t * 331.7 + 0.13, 1.0);
    const double th = 6.283185307179586 * fmod(t * 11.7, 1.0);
    const double vx = sp * cos(th), vy = sp * sin(th), w = 4.0 / 3.0 * eps / (1.0 - sp * sp), P = (eps - 1.0) / 3.0;
    const double ne = 1e-3 * sin(17.0 * t);
    return Moments{(float)(w - eps / 3.0 - 1.0), (float)(w * vx), (float)(w * vy), (float)(w * vx * vx + P + ne),
                   (float)(w * vx * vy + 0.5 * ne), (float)(w * vy * vy + P - ne)};
}

__device__ Out frame(Moments a, Moments b, int which) {
    const Frame<pf2> f = landau_fast<pf2>(pf2(1.0f), pf2(a.dE, b.dE), pf2(a.Mx, b.Mx), pf2(a.My, b.My),
                                          pf2(a.Sxx, b.Sxx), pf2(a.Sxy, b.Sxy), pf2(a.Syy, b.Syy));
    const pf2 v[7] = {f.ddelta_eps, f.eps, f.vx, f.vy, f.v2, f.g2, f.gamma};
    Out o;
    for (int k = 0; k < 7; ++k) o.f[k] = which ? v[k].v.y : v[k].v.x;
    return o;
}

__global__ void k_frames(int n, const Moments *in, Out *out, int *differ) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const Moments m = in[i], next = in[(i + 1) % n], rest{0, 0, 0, 0, 0, 0};
    const Out o = frame(m, m, 0), p[5] = {frame(m, m, 1), frame(m, next, 0), frame(next, m, 1), frame(m, rest, 0),
                                          frame(rest, m, 1)};
    out[i] = o;
    bool same = true;
    for (int k = 0; k < 5; ++k)
        for (int j = 0; j < 7; ++j) same = same && __float_as_int(p[k].f[j]) == __float_as_int(o.f[j]);
    if (!same) atomicAdd(differ, 1);
}

int main(int argc, char **argv) {
    if (argc != 3) return 2;
    const int n = 1 << 15;
    std::vector<Moments> h(n);
    for (int i = 0; i < n; ++i) h[i] = sample(i, n, std::atof(argv[1]), std::atof(argv[2]));
    Moments *d = nullptr;
    Out *dout = nullptr;
    int *dbad = nullptr, bad = 0;
    if (cudaMalloc(&d, sizeof(Moments) * n) != cudaSuccess || cudaMalloc(&dout, sizeof(Out) * n) != cudaSuccess ||
        cudaMalloc(&dbad, sizeof(int)) != cudaSuccess || cudaMemset(dbad, 0, sizeof(int)) != cudaSuccess)
        return 1;
    if (cudaMemcpy(d, h.data(), sizeof(Moments) * n, cudaMemcpyHostToDevice) != cudaSuccess) return 1;
    k_frames<<<n / 128, 128>>>(n, d, dout, dbad);
    std::vector<Out> out(n);
    if (cudaMemcpy(out.data(), dout, sizeof(Out) * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    if (cudaMemcpy(&bad, dbad, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    long double lean_v = 0, lean_d = 0;
    const float rest_a = (float)(4.0 / 3.0);  // the frame's own diagonal at rest
    for (int i = 0; i < n; ++i) {
        typedef long double L;
        const Moments m = h[i];
        const L a0 = (L)rest_a + m.dE, Mx = m.Mx, My = m.My;
        L delta = 0, vx = 0, vy = 0;
        for (int it = 0; it < 30; ++it) {
            const L xx = a0 - delta + m.Sxx, yy = a0 - delta + m.Syy, det = xx * yy - (L)m.Sxy * m.Sxy;
            vx = (yy * Mx - m.Sxy * My) / det;
            vy = (xx * My - m.Sxy * Mx) / det;
            delta -= (delta - (Mx * vx + My * vy)) / (1 - vx * vx - vy * vy);
        }
        const Out &o = out[i];
        lean_v += ((o.f[2] - vx) * vx + (o.f[3] - vy) * vy) / (vx * vx + vy * vy) / n;
        lean_d += (((L)m.dE - o.f[0]) / (Mx * o.f[2] + My * o.f[3]) - 1) / n;
    }
    std::printf("{\"differ\": %d, \"lean_v\": %.4e, \"lean_delta\": %.4e}\n", bad, (double)lean_v, (double)lean_d);
    return 0;
}
