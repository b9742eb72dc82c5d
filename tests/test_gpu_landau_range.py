"""The FP64 Landau frame at any reference energy: the problem is homogeneous,
so its accuracy must not depend on eps0, in the frame alone and in a whole
FP64 lattice."""
import json
import os
import subprocess

import numpy as np
import pytest

import workloads

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "numerics", "landau_range_check.cu")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("landau") / "check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-o", exe, SRC], check=True)
    return lambda *a: json.loads(subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                                text=True).stdout)


# Both solves end with the same few roundings: over the states of one eps0 the mean error may differ by a quarter and
# the largest by a factor of two, or by two units in the last place where the solve's own error is smaller than that.
# Speeds below, at and above the FP32 form's early exit, and beyond |v|^2 = 1/2, where the Newton solve takes over.
@pytest.mark.parametrize("vmax", [1e-4, 0.01, 0.3, 0.9])
@pytest.mark.parametrize("ring", [0, 1])
def test_frame_is_accurate_at_any_reference_energy(check, vmax, ring):
    unit = 2.0 ** -52
    for e, fast_max, fast_mean, solve_max, solve_mean in check(-38, 38, vmax, ring):
        assert fast_max <= max(2.0 * solve_max, 2 * unit), (e, fast_max, solve_max)
        assert fast_mean <= max(1.25 * solve_mean, unit), (e, fast_mean, solve_mean)


# far outside FP32's range too, and across the line to where only the Newton solve is left (a0 beyond 2^500, 3e150)
@pytest.mark.parametrize("lo,hi", [(-152, -148), (148, 152)])
def test_frame_beyond_fp32s_exponents(check, lo, hi):
    for e, fast_max, _, solve_max, _ in check(lo, hi, 0.3, 0):
        assert fast_max <= max(2.0 * solve_max, 2 * 2.0 ** -52), (e, fast_max, solve_max)


# A lattice's populations (deviations from rest) scale with eps0; 20 steps of a few roundings of 2^-53 each.
@pytest.mark.parametrize("stencil", ["sph26", "ring8"])
@pytest.mark.parametrize("eps0", [2e19, 1e-18])
def test_lattice_scales_with_its_reference_energy(stencil, eps0):
    nx, ny = 64, 48
    e, vx, vy = workloads.random_smooth(nx, ny, seed=6, deps=0.05, vmax=0.3)
    got = []
    for scale in (1.0, eps0):
        lat = rl.Lattice(nx, ny, 0.7, dtype="f64", eps0=scale, stencil=stencil,
                         forcing=dict(kmin=1, kmax=2, amp=1e-4, seed=5, redraw_period=8))
        lat.init_fields(e * scale, vx, vy)
        lat.step(20)
        m = lat.moments()
        got.append((lat.populations() / scale, m[0] / scale, m[1], m[2]))
        lat.close()
    for a, b in zip(*got):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.max(np.abs(a))
