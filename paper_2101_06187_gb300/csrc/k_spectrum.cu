// k_spectrum.cu -- the spectra of the velocity field (Sec. 4) in FP64.
//
// z = v_x + i v_y is transformed once (2D DFT); since every shell is
// symmetric under k -> -k, sum_shell |X|^2 + |Y|^2 = sum_shell |Z|^2 with X, Y
// the transforms of v_x, v_y, so E(n) = 1/2 sum_shell |Z|^2 / (nx ny)^2.
//
// One kernel transforms lines of any length up to 8192 in shared memory:
// Stockham passes of radix 8, 4, 2, 3, 5, 7 in registers, other prime factors
// by the symmetric direct sum.  It is bound by the FP64 pipe (2 per clock and
// SM on this GPU), so what counts is FP64 instructions: 34 per point of a 2048
// line instead of the 44 of radix-2 butterflies; a length with a factor 3 (the
// ensemble sides 384 and 768) no longer takes 4 n per point of a direct DFT.
// Only the modes asked for are finished: a line that needs 2K + 1 of its n
// outputs stops after the first passes and sums the rest directly where that
// is less work, and only the columns |kx| <= K are transformed at all.  The
// row pass reads the velocity arrays itself and the column pass sums |Z|^2
// into the shells (or the band) as the values come out, so nothing is packed
// or written back.
//
// Measured: moments, E(k) and the filtered velocity of a 2048^2 lattice 2.94 ->
// 2.06 ms; 100 steps and E(k) of 16 ensemble members with sides 256 to 1024
// 54.3 -> 13.9 ms (a 768^2 spectrum 11.6 ms of direct DFTs before).
#include <math.h>

#include <algorithm>

#include "rlbm_internal.h"

namespace rlbk {

namespace {

struct Z2 {
    double re, im;
};

__device__ __forceinline__ Z2 zadd(Z2 a, Z2 b) { return {a.re + b.re, a.im + b.im}; }
__device__ __forceinline__ Z2 zsub(Z2 a, Z2 b) { return {a.re - b.re, a.im - b.im}; }
__device__ __forceinline__ Z2 zmul(Z2 a, Z2 b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
__device__ __forceinline__ Z2 zload(const Z2 *p) {
    const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
    return {v.x, v.y};
}

// Forward twiddles w[k] = exp(-2 pi i k / n), k < n.
__global__ void k_dft_twiddles(Z2 *w, int n) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double s, c;
    sincospi(2.0 * (double)k / (double)n, &s, &c);
    w[k] = {c, -s};
}

// ---------------------------------------------------------------- line transform
constexpr int kMaxFactors = 16;

// Transform plan of lines of length n: the radices in pass order, the threads
// and lines of a block, and the passes actually run (the rest, if any, by the
// direct sum over the outputs wanted).
struct LinePlan {
    int n, nf, run, tpl, lpb;
    int f[kMaxFactors];
};

// Where line l starts and how far apart its elements are:
// (l % a) * s1 + (l / a) * s2 + j * es.
struct LineMap {
    int lines, a;
    long long s1, s2, es;
};

// The outputs wanted: all n, or the 2K + 1 frequencies |k| <= K.
struct Wanted {
    int all, K;
};

__device__ __forceinline__ void dft4(Z2 &a, Z2 &b, Z2 &c, Z2 &d) {
    const Z2 s = zadd(a, c), t = zsub(a, c), u = zadd(b, d), v = zsub(b, d);
    a = zadd(s, u);
    c = zsub(s, u);
    b = {t.re + v.im, t.im - v.re};  // t - i v
    d = {t.re - v.im, t.im + v.re};
}

template <int R>
__device__ __forceinline__ void dft(Z2 (&v)[R], const Z2 *w, int n) {
    if constexpr (R == 2) {
        const Z2 a = v[0], b = v[1];
        v[0] = zadd(a, b);
        v[1] = zsub(a, b);
    } else if constexpr (R == 4) {
        dft4(v[0], v[1], v[2], v[3]);
    } else if constexpr (R == 8) {
        Z2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
        dft4(e[0], e[1], e[2], e[3]);
        dft4(o[0], o[1], o[2], o[3]);
        const double h = 0.70710678118654752440;
        v[0] = zadd(e[0], o[0]);
        v[4] = zsub(e[0], o[0]);
        const Z2 p = {o[1].re + o[1].im, o[1].im - o[1].re};  // (1 - i) o1
        v[1] = {fma(h, p.re, e[1].re), fma(h, p.im, e[1].im)};
        v[5] = {fma(-h, p.re, e[1].re), fma(-h, p.im, e[1].im)};
        v[2] = {e[2].re + o[2].im, e[2].im - o[2].re};
        v[6] = {e[2].re - o[2].im, e[2].im + o[2].re};
        const Z2 q = {o[3].im - o[3].re, -(o[3].re + o[3].im)};  // (-1 - i) o3
        v[3] = {fma(h, q.re, e[3].re), fma(h, q.im, e[3].im)};
        v[7] = {fma(-h, q.re, e[3].re), fma(-h, q.im, e[3].im)};
    } else {  // odd R: pairs (s, R - s) share their sums and differences
        constexpr int H = (R - 1) / 2;
        Z2 c[H], S[H], D[H];
#pragma unroll
        for (int s = 0; s < H; ++s) {
            c[s] = zload(w + (s + 1) * (n / R));  // (cos, -sin)(2 pi (s + 1) / R)
            S[s] = zadd(v[s + 1], v[R - 1 - s]);
            D[s] = zsub(v[s + 1], v[R - 1 - s]);
        }
        const Z2 x0 = v[0];
#pragma unroll
        for (int s = 0; s < H; ++s) v[0] = zadd(v[0], S[s]);
#pragma unroll
        for (int k = 1; k <= H; ++k) {
            Z2 A = x0, B = {0.0, 0.0};
#pragma unroll
            for (int s = 1; s <= H; ++s) {
                const int m = (s * k) % R;
                const Z2 t = c[(m <= H ? m : R - m) - 1];
                const double sn = m <= H ? -t.im : t.im;
                A = {fma(t.re, S[s - 1].re, A.re), fma(t.re, S[s - 1].im, A.im)};
                B = {fma(sn, D[s - 1].re, B.re), fma(sn, D[s - 1].im, B.im)};
            }
            v[k] = {A.re + B.im, A.im - B.re};  // A - i B
            v[R - k] = {A.re - B.im, A.im + B.re};
        }
    }
}

// One Stockham pass of radix R over a line in place: butterfly i takes elements
// i + s n / R times w_{L R}^{s (i mod L)} and leaves the results at
// (i / L) L R + (i mod L) + s L.  tid: the thread within its line's tpl.
template <int R>
__device__ __forceinline__ void line_pass(int n, int L, int tpl, int tid, const Z2 *w, Z2 *sh) {
    constexpr int B = (8 + R - 1) / R;  // butterflies of a thread: tpl >= n / 8
    const int m = n / R, step = m / L;
    Z2 v[B][R];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int i = tid + b * tpl;
        if (i < m) {
            const int k = i % L;
#pragma unroll
            for (int s = 0; s < R; ++s) {
                v[b][s] = sh[i + s * m];
                if (s > 0 && L > 1) v[b][s] = zmul(v[b][s], zload(w + k * s * step));
            }
            dft<R>(v[b], w, n);
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int i = tid + b * tpl;
        if (i < m) {
            const int k = i % L, j = (i - k) * R + k;
#pragma unroll
            for (int s = 0; s < R; ++s) sh[j + s * L] = v[b][s];
        }
    }
}

// The odd radices out of line, so the registers they need are not taken from
// the power-of-two passes.
template <int R>
__device__ __noinline__ void odd_pass(int n, int L, int tpl, int tid, const Z2 *w, Z2 *sh) {
    line_pass<R>(n, L, tpl, tid, w, sh);
}

// The same for a prime radix R > 7: sums and differences of the twiddled
// pairs (s, R - s) in place, then outputs t and R - t of a butterfly as two
// real-coefficient sums over the (R - 1) / 2 pairs (a quarter of the direct
// DFT's multiply-adds).
__device__ __noinline__ void prime_pass(int n, int R, int L, int tpl, int tid, const Z2 *w, Z2 *sh) {
    const int m = n / R, step = m / L, H = (R - 1) / 2;
    for (int u = tid; u < m * H; u += tpl) {
        const int i = u % m, s = u / m + 1, k = i % L;
        Z2 a = sh[i + s * m], b = sh[i + (R - s) * m];
        if (L > 1) {
            a = zmul(a, zload(w + k * s * step));
            b = zmul(b, zload(w + k * (R - s) * step));
        }
        sh[i + s * m] = zadd(a, b);
        sh[i + (R - s) * m] = zsub(a, b);
    }
    __syncthreads();
    constexpr int B = 5;  // m (R + 1) / 2 items over tpl >= n / 8 threads
    Z2 lo[B], hi[B];
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int u = tid + b * tpl;
        if (u < m * (H + 1)) {
            const int i = u % m, t = u / m;
            Z2 A = sh[i], D = {0.0, 0.0};
            int idx = 0;  // s t mod R
            for (int s = 1; s <= H; ++s) {
                idx += t;
                if (idx >= R) idx -= R;
                const Z2 c = zload(w + idx * m);  // (cos, -sin)(2 pi s t / R)
                const Z2 sum = sh[i + s * m], dif = sh[i + (R - s) * m];
                A = {fma(c.re, sum.re, A.re), fma(c.re, sum.im, A.im)};
                D = {fma(-c.im, dif.re, D.re), fma(-c.im, dif.im, D.im)};
            }
            lo[b] = {A.re + D.im, A.im - D.re};
            hi[b] = {A.re - D.im, A.im + D.re};
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int u = tid + b * tpl;
        if (u < m * (H + 1)) {
            const int i = u % m, t = u / m, k = i % L, j = (i - k) * R + k;
            sh[j + t * L] = lo[b];
            if (t > 0) sh[j + (R - t) * L] = hi[b];
        }
    }
}

// A block's lines, one per tpl threads (every thread of the block takes part
// in the waits): `load(j)` an input element, `emit(f, z)` takes output
// frequency f (0 <= f < n) where `want` has it.  Starts and ends with the
// line's shared memory free.
template <typename Load, typename Emit>
__device__ __forceinline__ void transform_line(const LinePlan &pl, const Z2 *w, Z2 *sh, int tid, bool live,
                                               const Wanted &want, Load &&load, Emit &&emit) {
    const int n = pl.n, tpl = pl.tpl;
    for (int j = tid; j < n; j += tpl) sh[j] = live ? load(j) : Z2{0.0, 0.0};
    __syncthreads();
    int L = 1;
    for (int q = 0; q < pl.run; ++q) {
        const int R = pl.f[q];
        switch (R) {
        case 8: line_pass<8>(n, L, tpl, tid, w, sh); break;
        case 4: line_pass<4>(n, L, tpl, tid, w, sh); break;
        case 2: line_pass<2>(n, L, tpl, tid, w, sh); break;
        case 3: odd_pass<3>(n, L, tpl, tid, w, sh); break;
        case 5: odd_pass<5>(n, L, tpl, tid, w, sh); break;
        case 7: odd_pass<7>(n, L, tpl, tid, w, sh); break;
        default: prime_pass(n, R, L, tpl, tid, w, sh);
        }
        __syncthreads();
        L *= R;
    }
    // the outputs wanted: X[f] = sum_g w_n^{g f} Y_g[f mod L] over the n / L sub-transforms of length L (one, the
    // transform itself, where every pass was run)
    const int S = want.all ? n : 2 * want.K + 1;
    for (int u = tid; u < S; u += tpl) {
        const int f = want.all || u <= want.K ? u : n - S + u, kap = f % L;
        Z2 acc = sh[kap];
        int idx = 0;
        for (int g = 1; g < n / L; ++g) {
            idx += f;
            if (idx >= n) idx -= n;
            const Z2 c = zload(w + idx), y = sh[g * L + kap];
            acc = {fma(y.re, c.re, fma(-y.im, c.im, acc.re)), fma(y.re, c.im, fma(y.im, c.re, acc.im))};
        }
        if (live) emit(f, acc);
    }
    __syncthreads();
}

// T: the most threads of a block (256, or 1024 for lines above 2048, where a
// thread has 64 registers and some of its values spill).
#define RLBM_FFT_BOUNDS __launch_bounds__(T, T == 256 ? 2 : 1)

// Rows of (vx, vy) -> z[line][f] for the wanted f.
template <int T>
__global__ void RLBM_FFT_BOUNDS k_fft_rows(LinePlan pl, int lines, const double *__restrict__ vx,
                                                   const double *__restrict__ vy, Z2 *__restrict__ z, Wanted want,
                                                   const Z2 *__restrict__ w) {
    extern __shared__ Z2 sh_all[];
    const int sub = threadIdx.x / pl.tpl, tid = threadIdx.x - sub * pl.tpl;
    const int line = blockIdx.x * pl.lpb + sub;
    const long long base = (long long)line * pl.n;
    transform_line(
        pl, w, sh_all + (long long)sub * pl.n, tid, line < lines, want,
        [&](int j) { return Z2{__ldg(vx + base + j), __ldg(vy + base + j)}; },
        [&](int f, Z2 v) { z[base + f] = v; });
}

// Lines of z in place (the 3D transforms).
template <int T>
__global__ void RLBM_FFT_BOUNDS k_fft_inplace(LinePlan pl, LineMap m, Z2 *z, const Z2 *__restrict__ w) {
    extern __shared__ Z2 sh_all[];
    const int sub = threadIdx.x / pl.tpl, tid = threadIdx.x - sub * pl.tpl;
    const int line = blockIdx.x * pl.lpb + sub;
    Z2 *const p = z + (line % m.a) * m.s1 + (line / m.a) * m.s2;
    transform_line(
        pl, w, sh_all + (long long)sub * pl.n, tid, line < m.lines, Wanted{1, 0}, [&](int j) { return p[j * m.es]; },
        [&](int f, Z2 v) { p[f * m.es] = v; });
}

__device__ __forceinline__ int signed_k(int j, int n) { return (j < (n + 1) / 2) ? j : j - n; }

// The shell n of |k|^2 = k2: |k| in [n - 1/2, n + 1/2), i.e. n^2 - n < k2 <= n^2 + n
// (in integers, |k_a| <= 4096; the square root only guesses n).
__device__ __forceinline__ int shell_of(int k2) {
    int n = (int)(sqrtf((float)k2) + 0.5f);
    while (n * n + n < k2) ++n;
    while (n > 0 && n * n - n >= k2) --n;
    return n;
}

// Columns of z (the kx wanted) -> scale * sum |Z|^2 per shell (BAND = false:
// shells below nshells into out[]) or over |k|^2 < kf2 (BAND: into out[0]).
// Blocks walk the columns with a stride, so each adds its sums to out once.
template <bool BAND, int T>
__global__ void RLBM_FFT_BOUNDS k_fft_columns(LinePlan pl, int cols, int nx, const Z2 *__restrict__ z,
                                                      Wanted want, const Z2 *__restrict__ w, int nshells, double kf2,
                                                      double scale, double *out) {
    extern __shared__ Z2 sh_all[];
    double *hist = reinterpret_cast<double *>(sh_all + (long long)pl.lpb * pl.n);
    const int bins = BAND ? 1 : nshells;
    for (int i = threadIdx.x; i < bins; i += blockDim.x) hist[i] = 0.0;
    __syncthreads();
    const int sub = threadIdx.x / pl.tpl, tid = threadIdx.x - sub * pl.tpl;
    double band = 0.0;
    for (int c0 = blockIdx.x * pl.lpb; c0 < cols; c0 += gridDim.x * pl.lpb) {
        const int c = c0 + sub;  // the columns 0 .. Kx and nx - Kx .. nx - 1, or all
        const int jx = (cols == nx || 2 * c < cols) ? c : nx - cols + c;
        const int kx = signed_k(jx, nx);
        transform_line(
            pl, w, sh_all + (long long)sub * pl.n, tid, c < cols, want,
            [&](int j) { return zload(z + ((long long)j * nx + jx)); },
            [&](int f, Z2 v) {
                const int ky = signed_k(f, pl.n), k2 = kx * kx + ky * ky;
                const double e = v.re * v.re + v.im * v.im;
                if constexpr (BAND) {
                    if ((double)k2 < kf2) band += e;
                } else {
                    const int s = shell_of(k2);
                    if (s < nshells) atomicAdd(&hist[s], e);
                }
            });
    }
    if constexpr (BAND) {
        for (int o = 16; o > 0; o >>= 1) band += __shfl_down_sync(0xffffffffu, band, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&hist[0], band);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < bins; i += blockDim.x)
        if (hist[i] != 0.0) atomicAdd(&out[i], scale * hist[i]);
}

// Per-shell running sums of E and E^2 for time statistics of the spectrum.
__global__ void k_accumulate(const double *E, int n, double *sum, double *sq) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        sum[i] += E[i];
        sq[i] += E[i] * E[i];
    }
}

// ---------------------------------------------------------------- plans and launches
// FP64 operations per point of a pass (rough), by radix.
double pass_cost(int r, bool first) {
    const double tw = first ? 0.0 : 4.0 * (r - 1) / r;
    switch (r) {
    case 8: return 6.5 + tw;
    case 4: return 4.0 + tw;
    case 2: return 2.0 + tw;
    default: return r + 1.0 + tw;
    }
}

// Plan for `lines` lines of length n of which `wanted` outputs are needed.
LinePlan make_plan(int n, int lines, int wanted) {
    LinePlan p{};
    p.n = n;
    int m = n;
    auto take = [&](int r) {
        while (m % r == 0) {
            p.f[p.nf++] = r;
            m /= r;
        }
    };
    for (int r : {8, 4, 2, 3, 5, 7}) take(r);
    for (int r = 11; m > 1; r += 2) {
        if ((long long)r * r > m) r = m;  // what is left is prime
        take(r);
    }
    if (p.nf == 0) p.f[p.nf++] = 1;  // n = 1: not a lattice, kept well defined
    // threads of a line: at least n / 8 (a thread holds 8 values), in whole warps; several short lines share
    // a block where there are enough of them for every SM to have two blocks
    p.tpl = std::min(1024, ((n + 7) / 8 + 31) & ~31);
    p.lpb = std::max(1, std::min(256 / p.tpl, lines / 304));
    // passes to run before the direct sum over the outputs wanted, if that is less work
    double spent = 0.0, best = 1e300;
    int L = 1;
    p.run = p.nf;
    for (int q = 0; q < p.nf; ++q) {
        spent += pass_cost(p.f[q], q == 0);
        L *= p.f[q];
        const double c = spent + (q + 1 < p.nf ? 4.0 * std::max(wanted, p.tpl / 4) / L : 0.0);
        if (c < best) {
            best = c;
            p.run = q + 1;
        }
    }
    return p;
}

// The most shared memory a legal call asks for: one line of 8192 and 4096
// shells.  A kernel's limit is shared by all handles and host threads, so it is
// only ever set to this: set to a call's own size, another thread's smaller
// call could lower it before the launch, which then failed.
constexpr int kMostSmem = 8192 * (int)sizeof(Z2) + 4096 * (int)sizeof(double);

template <typename Kernel, typename... Args>
cudaError_t launch(Kernel kernel, int blocks, int threads, size_t smem, cudaStream_t s, Args... args) {
    if (smem > 48 * 1024) {  // what every kernel may use without asking
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMostSmem);
        if (e != cudaSuccess) return e;
    }
    kernel<<<blocks, threads, smem, s>>>(args...);
    return cudaGetLastError();
}

size_t line_smem(const LinePlan &p) { return (size_t)p.lpb * p.n * sizeof(Z2); }

// Transform of (vx, vy) and the sum of scale |Z|^2 over shells or a band.
template <bool BAND>
cudaError_t transform_2d(const double *vx, const double *vy, int nx, int ny, int K, int nshells, double kf2,
                         double scale, double *work, double *out, cudaStream_t s) {
    Z2 *z = reinterpret_cast<Z2 *>(work), *wx = z + (size_t)nx * ny, *wy = wx + nx;
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * (BAND ? 1 : nshells), s);
    if (e != cudaSuccess || K < 0) return e;  // no mode asked for
    auto wanted = [&](int n) { return 2ll * K + 1 >= n ? Wanted{1, n} : Wanted{0, K}; };
    const Wanted wr = wanted(nx), wc = wanted(ny);
    const int cols = wr.all ? nx : 2 * K + 1;
    const LinePlan pr = make_plan(nx, ny, cols), pc = make_plan(ny, cols, wc.all ? ny : 2 * K + 1);
    const int tr = pr.tpl * pr.lpb, tc = pc.tpl * pc.lpb;
    e = launch(tr <= 256 ? k_fft_rows<256> : k_fft_rows<1024>, (ny + pr.lpb - 1) / pr.lpb, tr, line_smem(pr), s, pr, ny,
               vx, vy, z, wr, (const Z2 *)wx);
    if (e != cudaSuccess) return e;
    // as many blocks as the GPU holds (128 registers a thread below 256 threads): each adds its sums once
    const size_t smem = line_smem(pc) + sizeof(double) * (BAND ? 1 : nshells);
    const int per_sm = std::max(1, (int)std::min((size_t)(512 / tc), (size_t)(227 * 1024) / (smem + 1024)));
    return launch(tc <= 256 ? k_fft_columns<BAND, 256> : k_fft_columns<BAND, 1024>,
                  std::min((cols + pc.lpb - 1) / pc.lpb, 152 * per_sm), tc, smem, s, pc, cols, nx, (const Z2 *)z, wc,
                  (const Z2 *)wy, nshells, kf2, scale, out);
}

}  // namespace

cudaError_t launch_accumulate(const double *E, int n, double *sum, double *sq, cudaStream_t s) {
    k_accumulate<<<(n + 255) / 256, 256, 0, s>>>(E, n, sum, sq);
    return cudaGetLastError();
}

size_t spectrum_work_doubles(int nx, int ny) { return 2 * ((size_t)nx * ny + (size_t)nx + (size_t)ny); }

size_t spectrum_work_doubles3(int nx, int ny, int nz) {
    return 2 * (2 * (size_t)nx * ny * nz + (size_t)nx + (size_t)ny + (size_t)nz);
}

// The twiddle tables at the end of a work area (2D: nz = 0), filled once.
cudaError_t launch_spectrum_tables(int nx, int ny, int nz, double *work, cudaStream_t s) {
    Z2 *w = reinterpret_cast<Z2 *>(work) + (nz ? 2 * (size_t)nx * ny * nz : (size_t)nx * ny);
    for (int n : {nx, ny, nz}) {
        if (n > 0) k_dft_twiddles<<<(n + 255) / 256, 256, 0, s>>>(w, n);
        w += n;
    }
    return cudaGetLastError();
}

// Mean square of the velocity with every mode |k| >= kf removed:
// <|v_f|^2> = sum_{|k| < kf} |v_hat(k)|^2 = sum_{|k| < kf} |Z(k)|^2 / (nx ny)^2
// (the set |k| < kf is symmetric under k -> -k, as for the shells).
cudaError_t launch_band_power(const double *vx, const double *vy, int nx, int ny, double kf, double *work,
                              double *out, cudaStream_t s) {
    const double count = (double)nx * ny;
    const int K = kf > 16384.0 ? 16384 : (int)ceil(kf) - 1;  // the largest |kx| below kf
    return transform_2d<true>(vx, vy, nx, ny, K, 0, kf * kf, 1.0 / (count * count), work, out, s);
}

cudaError_t launch_spectrum(const double *vx, const double *vy, int nx, int ny, int nshells, double *work,
                            double *Ek, cudaStream_t s) {
    const double count = (double)nx * ny;
    // shell n holds |k| >= n - 1/2 and |k| >= |kx|
    return transform_2d<false>(vx, vy, nx, ny, nshells - 1, nshells, 0.0, 0.5 / (count * count), work, Ek, s);
}

// ---------------------------------------------------------------- 3D spectra
// The three velocity components as two complex fields Z1 = vx + i vy and
// Z2 = vz, each transformed along x, y and z; over a shell (symmetric under
// k -> -k) the sum of |Z1|^2 + |Z2|^2 is the sum of |v_hat_x|^2 + |v_hat_y|^2
// + |v_hat_z|^2, times vol^2.
namespace {

__global__ void k_pack_z3(const double *vx, const double *vy, const double *vz, Z2 *z1, Z2 *z2, long long count) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) {
        z1[i] = {vx[i], vy[i]};
        z2[i] = {vz[i], 0.0};
    }
}

__device__ __forceinline__ int mode_k2(long long i, int nx, int ny, int nz) {
    const int jx = (int)(i % nx), jy = (int)((i / nx) % ny), jz = (int)(i / ((long long)nx * ny));
    const int kx = signed_k(jx, nx), ky = signed_k(jy, ny), kz = signed_k(jz, nz);
    return kx * kx + ky * ky + kz * kz;
}

__global__ void k_shell_bin3(const Z2 *z1, const Z2 *z2, int nx, int ny, int nz, int nshells, double scale,
                             double *Ek) {
    extern __shared__ double hist[];
    for (int i = threadIdx.x; i < nshells; i += blockDim.x) hist[i] = 0.0;
    __syncthreads();
    const long long count = (long long)nx * ny * nz;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x) {
        const int sh = shell_of(mode_k2(i, nx, ny, nz));
        if (sh < nshells)
            atomicAdd(&hist[sh], z1[i].re * z1[i].re + z1[i].im * z1[i].im + z2[i].re * z2[i].re + z2[i].im * z2[i].im);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nshells; i += blockDim.x)
        if (hist[i] != 0.0) atomicAdd(&Ek[i], scale * hist[i]);
}

__global__ void k_band_sum3(const Z2 *z1, const Z2 *z2, int nx, int ny, int nz, double kf2, double scale,
                            double *out) {
    __shared__ double red[256];
    double acc = 0.0;
    const long long count = (long long)nx * ny * nz;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (long long)gridDim.x * blockDim.x)
        if ((double)mode_k2(i, nx, ny, nz) < kf2)
            acc += z1[i].re * z1[i].re + z1[i].im * z1[i].im + z2[i].re * z2[i].re + z2[i].im * z2[i].im;
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out, scale * red[0]);
}

cudaError_t lines_inplace(Z2 *z, int n, const LineMap &m, const Z2 *w, cudaStream_t s) {
    const LinePlan p = make_plan(n, m.lines, n);
    const int t = p.tpl * p.lpb;
    return launch(t <= 256 ? k_fft_inplace<256> : k_fft_inplace<1024>, (m.lines + p.lpb - 1) / p.lpb, t, line_smem(p), s,
                  p, m, z, w);
}

cudaError_t transform_3d(const double *vx, const double *vy, const double *vz, int nx, int ny, int nz, double *work,
                         cudaStream_t s) {
    const long long count = (long long)nx * ny * nz, slab = (long long)nx * ny;
    Z2 *z1 = reinterpret_cast<Z2 *>(work), *z2 = z1 + count;
    const Z2 *w = z2 + count;
    k_pack_z3<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(vx, vy, vz, z1, z2, count);
    cudaError_t e = cudaGetLastError();
    for (Z2 *z : {z1, z2}) {
        if (e == cudaSuccess) e = lines_inplace(z, nx, LineMap{ny * nz, ny * nz, nx, 0, 1}, w, s);
        if (e == cudaSuccess) e = lines_inplace(z, ny, LineMap{nx * nz, nx, 1, slab, nx}, w + nx, s);
        if (e == cudaSuccess) e = lines_inplace(z, nz, LineMap{(int)slab, (int)slab, 1, 0, slab}, w + nx + ny, s);
    }
    return e;
}

}  // namespace

cudaError_t launch_spectrum3(const double *vx, const double *vy, const double *vz, int nx, int ny, int nz, int nshells,
                             double *work, double *Ek, cudaStream_t s) {
    const long long count = (long long)nx * ny * nz;
    cudaError_t e = transform_3d(vx, vy, vz, nx, ny, nz, work, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(Ek, 0, sizeof(double) * nshells, s);
    if (e != cudaSuccess) return e;
    const Z2 *z1 = reinterpret_cast<const Z2 *>(work);
    k_shell_bin3<<<304, 256, sizeof(double) * nshells, s>>>(z1, z1 + count, nx, ny, nz, nshells,
                                                            0.5 / ((double)count * (double)count), Ek);
    return cudaGetLastError();
}

cudaError_t launch_band_power3(const double *vx, const double *vy, const double *vz, int nx, int ny, int nz, double kf,
                               double *work, double *out, cudaStream_t s) {
    const long long count = (long long)nx * ny * nz;
    cudaError_t e = transform_3d(vx, vy, vz, nx, ny, nz, work, s);
    if (e != cudaSuccess) return e;
    e = cudaMemsetAsync(out, 0, sizeof(double), s);
    if (e != cudaSuccess) return e;
    const Z2 *z1 = reinterpret_cast<const Z2 *>(work);
    k_band_sum3<<<304, 256, 0, s>>>(z1, z1 + count, nx, ny, nz, kf * kf, 1.0 / ((double)count * (double)count), out);
    return cudaGetLastError();
}

}  // namespace rlbk
