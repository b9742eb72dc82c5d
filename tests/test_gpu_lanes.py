"""Results of the FP32 form do not depend on which nodes a kernel packs into
one thread: the frame of a lane is its own, so the one-column kernel (rows y,
y + 1) equals the packed one (columns x, x + 1) bit for bit, and slabs of any
height the whole lattice, also where some nodes pass the frame's early exit
and their partners do not (|v| around 0.05)."""
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
from paper_2101_06187_gb300 import slab  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
FORCING = dict(kmin=1, kmax=3, amp=2e-4, seed=31, redraw_period=5)


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("lanes") / "check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-o", exe, os.path.join(HERE, "numerics", "landau_lanes_check.cu")],
                   check=True)
    return lambda *a: json.loads(subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                                text=True).stdout)


@pytest.mark.parametrize("lo,hi", [(0.0, 0.04), (0.03, 0.06), (0.05, 0.08), (0.05, 0.3), (0.0, 0.95)])
def test_a_lanes_frame_is_its_own(check, lo, hi):
    assert check(lo, hi)["differ"] == 0


def _run(kernel, nx, ny, fields, **kw):
    lat = rl.Lattice(nx, ny, 0.6, dtype="f32", forcing=FORCING, kernel=kernel, **kw)
    lat.init_fields(*fields)
    lat.step(12)
    f = lat.populations()
    lat.close()
    return f


@pytest.mark.parametrize("size", [(32, 41), (66, 40), (128, 33)])
@pytest.mark.parametrize("kw", [{}, dict(cfl=0.625), dict(cfl=0.5, eta_s=0.02, dt=0.05)])
@pytest.mark.parametrize("vmax", [0.12, 0.3])
def test_one_column_kernel_equals_packed_bitwise(size, kw, vmax):
    fields = workloads.random_smooth(*size, seed=sum(size), vmax=vmax)
    np.testing.assert_array_equal(_run("gather", *size, fields, **kw), _run("packed", *size, fields, **kw))


# odd heights and offsets, one and two halo rows; "auto" is the untuned default
@pytest.mark.parametrize("world,halo,kernel", [(2, 1, "auto"), (3, 1, "auto"), (3, 2, "auto"), (3, 1, "gather"),
                                               (3, 1, "packed"), (3, 2, "fused2")])
@pytest.mark.parametrize("vmax", [0.12, 0.3])
def test_slabs_equal_the_whole_lattice_across_the_early_exit(world, halo, kernel, vmax):
    nx, ny, tau, nsteps = 64, 67, 0.6, 24
    fields = workloads.random_smooth(nx, ny, seed=8, deps=0.05, vmax=vmax)
    speed = np.hypot(fields[1], fields[2])
    assert speed.min() < 0.04 and speed.max() > 0.056
    whole = rl.Lattice(nx, ny, tau, dtype="f32", forcing=FORCING, kernel=kernel)
    whole.init_fields(*fields)
    whole.step(nsteps)
    ref = whole.populations()
    whole.close()
    group = slab.SlabGroup(nx, ny, tau, world, halo, dtype="f32", forcing=FORCING, kernel=kernel)
    group.init_fields(*fields)
    group.step(nsteps)
    got = np.concatenate([s.lat.populations()[:, slice(*s.rows.interior), :] for s in group.slabs], axis=1)
    group.close()
    np.testing.assert_array_equal(got, ref)
