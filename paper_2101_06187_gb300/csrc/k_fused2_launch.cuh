// k_fused2_launch.cuh -- host-side launch templates of the two-steps-per-
// launch kernels (k_step_fused2.cuh), shared by the translation units that
// instantiate them for each streaming mode.
#pragma once

#include "k_step_fused2.cuh"
#include "rlbm_internal.h"

namespace rlbk {

// Tile shape: output tile TW x TH, NT threads, MINB resident CTAs per SM
// (shared memory per CTA: 17 (TW + 4)(TH + 2) stored values); SM is the
// streaming mode of the single-lattice kernels.
template <typename TS, int TW, int TH, int NT, int MINB, int SM>
struct Fused2 {
    static constexpr int smem = fused2_smem_bytes<TS, TW, TH>();

    template <bool FORCED, typename I>
    static void *fn() {
        return reinterpret_cast<void *>(&k_step_fused2<TS, FORCED, TW, TH, NT, MINB, I, SM>);
    }
    static cudaError_t set_smem(void *f) {
        return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    }
    static cudaError_t prepare() {
        for (void *f : {fn<true, int>(), fn<false, int>(), fn<true, long long>(), fn<false, long long>()}) {
            const cudaError_t e = set_smem(f);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    static cudaError_t launch(bool forced, const void *qin, void *qout, const void *F, const StepParams &p,
                              cudaStream_t s) {
        const TS *in = static_cast<const TS *>(qin);
        TS *out = static_cast<TS *>(qout);
        const float *f = static_cast<const float *>(F);
        const dim3 grid((p.nx + TW - 1) / TW, (p.ny + TH - 1) / TH, 1);
        const bool idx32 = (long long)NC * p.plane < (1ll << 31) - 1;
        if (idx32) {
            if (forced) k_step_fused2<TS, true, TW, TH, NT, MINB, int, SM><<<grid, NT, smem, s>>>(in, out, f, p);
            else k_step_fused2<TS, false, TW, TH, NT, MINB, int, SM><<<grid, NT, smem, s>>>(in, out, f, p);
        } else {
            if (forced) k_step_fused2<TS, true, TW, TH, NT, MINB, long long, SM><<<grid, NT, smem, s>>>(in, out, f, p);
            else k_step_fused2<TS, false, TW, TH, NT, MINB, long long, SM><<<grid, NT, smem, s>>>(in, out, f, p);
        }
        return cudaGetLastError();
    }
};

// The tile shapes on offer, by (bx, by) = (TW, TH) of the launch shape:
// X(TW, TH, threads of the FP32 single-lattice kernels, threads of the
// 16-bit and ensemble kernels, resident CTAs).  The FP32 body fits 96
// registers, so 20 warps an SM instead of 16 hide more of the loads (64 x 8:
// 59.3 -> 61.2 GLUPS at 4096^2, 50.4 -> 51.0 at 1024^2, 128 -> 160 threads;
// 64 x 16: 54.9 -> 58.4 and 46.4 -> 49.3, 256 -> 320; 128 x 8: 56.1 -> 57.6;
// 32 x 16: 54.6 -> 56.0).  More warps spill (64 x 8 at 4 x 192: 45.8 at 1024^2) or
// leave a tile too few threads (5 x 96: 55.6 at 4096^2); the ensemble body
// spills at 96 registers (16 fields: 13.9 -> 14.6 ms) and stays at 128.
#define RLBM_FUSED2_SHAPES(X) \
    X(64, 16, 320, 256, 2)    \
    X(64, 8, 160, 128, 4)     \
    X(32, 16, 160, 128, 4)    \
    X(128, 8, 320, 256, 2)

// A 64 x 8 launch of few tiles has SMs with one or two blocks, whose time is
// the chain of a thread's node pairs (340 of the first step, 256 of the second), not
// occupancy.  Up to one tile for each of the 152 SMs: 352 threads, one pair
// each per step (256^2: 2.43 us per step against 2.98 with 128 threads, 2.69
// with 256, 3.15 with 160).  Up to two: 256 threads (384^2: 3.74 us against
// 3.83, 4.34 with 352, 3.98 with 160).  Beyond, 160 (512 x 384: 4.84 against
// 4.92 with 128, 5.39 with 256).
constexpr int kOneTile = 152, kOneTileThreads = 352;
constexpr int kTwoTiles = 2 * 152, kTwoTilesThreads = 256;

// Below cfl 1 the weights of the launch take registers too: the four-CTA shapes
// spill in 96 and keep the other threads (64 x 8 at cfl 0.625: 21.8 us per step
// with 128 at 1024^2 against 23.3 with 160, 288 against 303 at 4096^2); the
// two-CTA shapes lose more by fewer warps (64 x 16: 23.3 with 256, 22.5 with 320).
template <typename TS, int NT32, int NT, int MB, int SM>
constexpr int fused2_threads() {
    return std::is_same<TS, float>::value && !(SM == kStreamSub1 && MB == 4) ? NT32 : NT;
}

template <typename TS, int SM>
cudaError_t fused2_prepare_t() {
#define X(TW, TH, NT32, NT, MB)                                                                      \
    {                                                                                                \
        const cudaError_t e = Fused2<TS, TW, TH, fused2_threads<TS, NT32, NT, MB, SM>(), MB, SM>::prepare(); \
        if (e != cudaSuccess) return e;                                                              \
    }
    RLBM_FUSED2_SHAPES(X)
#undef X
    if constexpr (std::is_same<TS, float>::value) {
        const cudaError_t e = Fused2<TS, 64, 8, kOneTileThreads, 1, SM>::prepare();
        return e != cudaSuccess ? e : Fused2<TS, 64, 8, kTwoTilesThreads, 2, SM>::prepare();
    }
    return cudaSuccess;
}

template <typename TS, int SM>
cudaError_t fused2_launch_t(const LaunchCfg &cfg, bool forced, const void *qin, void *qout, const void *F,
                            const StepParams &p, cudaStream_t s) {
    if constexpr (std::is_same<TS, float>::value) {
        const long long tiles = (long long)((p.nx + 63) / 64) * ((p.ny + 7) / 8);
        if (cfg.bx == 64 && cfg.by == 8 && tiles <= kOneTile)
            return Fused2<TS, 64, 8, kOneTileThreads, 1, SM>::launch(forced, qin, qout, F, p, s);
        if (cfg.bx == 64 && cfg.by == 8 && tiles <= kTwoTiles)
            return Fused2<TS, 64, 8, kTwoTilesThreads, 2, SM>::launch(forced, qin, qout, F, p, s);
    }
#define X(TW, TH, NT32, NT, MB)                                                                        \
    if (cfg.bx == TW && cfg.by == TH)                                                                  \
        return Fused2<TS, TW, TH, fused2_threads<TS, NT32, NT, MB, SM>(), MB, SM>::launch(forced, qin, qout, F, p, s);
    RLBM_FUSED2_SHAPES(X)
#undef X
    return cudaErrorInvalidConfiguration;
}

// The ensemble kernels of tile shape TW x TH (CFL 1).
template <typename TS, int TW, int TH, int NT, int MINB>
struct Fused2Batch {
    static constexpr int smem = fused2_smem_bytes<TS, TW, TH>();
    static cudaError_t prepare() {
        for (void *f : {reinterpret_cast<void *>(&k_step_batch_fused2<TS, TW, TH, NT, MINB, true>),
                        reinterpret_cast<void *>(&k_step_batch_fused2<TS, TW, TH, NT, MINB, false>)}) {
            const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    }
    static cudaError_t launch(int grid, const void *runs, int nruns, int ntiles, int two, cudaStream_t s) {
        const BatchRun *r = static_cast<const BatchRun *>(runs);
        if (two) k_step_batch_fused2<TS, TW, TH, NT, MINB, true><<<grid, NT, smem, s>>>(r, nruns, ntiles);
        else k_step_batch_fused2<TS, TW, TH, NT, MINB, false><<<grid, NT, smem, s>>>(r, nruns, ntiles);
        return cudaGetLastError();
    }
};

template <typename TS>
cudaError_t batch_prepare_t() {
#define X(TW, TH, NT32, NT, MB)                                                  \
    {                                                                      \
        const cudaError_t e = Fused2Batch<TS, TW, TH, NT, MB>::prepare();  \
        if (e != cudaSuccess) return e;                                    \
    }
    RLBM_FUSED2_SHAPES(X)
#undef X
    return cudaSuccess;
}

template <typename TS>
cudaError_t batch_launch_t(const LaunchCfg &cfg, int grid, const void *runs, int nruns, int ntiles, int two,
                           cudaStream_t s) {
#define X(TW, TH, NT32, NT, MB)                                                                       \
    if (cfg.bx == TW && cfg.by == TH)                                                           \
        return Fused2Batch<TS, TW, TH, NT, MB>::launch(grid, runs, nruns, ntiles, two, s);
    RLBM_FUSED2_SHAPES(X)
#undef X
    return cudaErrorInvalidConfiguration;
}

// Per storage type and streaming mode, one translation unit each
// (k_fused2_inst.cuh), so the many kernel instantiations compile in
// parallel: the single-lattice kernels at CFL 1 with the ensemble kernels,
// and the single-lattice kernels at 0 < cfl < 1.
#define RLBM_FUSED2_TYPE_ENTRIES(SFX)                                                                          \
    cudaError_t fused2_prepare_cfl1_##SFX();                                                                   \
    cudaError_t fused2_launch_cfl1_##SFX(const LaunchCfg &cfg, bool forced, const void *qin, void *qout,        \
                                         const void *F, const StepParams &p, cudaStream_t s);                  \
    cudaError_t fused2_launch_batch_##SFX(const LaunchCfg &cfg, int grid, const void *runs, int nruns,         \
                                          int ntiles, int two, cudaStream_t s);                                \
    cudaError_t fused2_prepare_sub1_##SFX();                                                                   \
    cudaError_t fused2_launch_sub1_##SFX(const LaunchCfg &cfg, bool forced, const void *qin, void *qout,        \
                                         const void *F, const StepParams &p, cudaStream_t s);
RLBM_FUSED2_TYPE_ENTRIES(f32)
RLBM_FUSED2_TYPE_ENTRIES(bf16)
RLBM_FUSED2_TYPE_ENTRIES(f16)
#undef RLBM_FUSED2_TYPE_ENTRIES

}  // namespace rlbk
