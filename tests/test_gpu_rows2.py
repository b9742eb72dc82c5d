"""RLBM_KERNEL_GATHER of FP32 storage: two rows a thread in packed lanes at
cfl <= 1, one node a thread above.  Where nx is even it equals the packed
kernel bit for bit; odd sides are compared with the oracle."""
import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

FORCING = dict(kmin=1, kmax=1, amp=1e-4, seed=3, redraw_period=7)


def _run(kernel, nx, ny, fields, forcing, block=None, **kw):
    lat = rl.Lattice(nx, ny, 0.6, dtype="f32", forcing=forcing, kernel=kernel, **kw)
    if block:
        lat.set_launch(kernel, *block, 1)
    lat.init_fields(*fields)
    for n in (2, 5, 6):
        lat.step(n)
    f = lat.populations()
    lat.close()
    return f


# odd and even ny (an odd last row is updated alone), the 4 x 4 minimum, edges of the blocks
@pytest.mark.parametrize("size", [(4, 4), (6, 5), (66, 41), (30, 131), (258, 16)])
@pytest.mark.parametrize("kw", [{}, dict(cfl=0.625), dict(cfl=0.5, eta_s=0.02, dt=0.05), dict(cfl=1.25)])
@pytest.mark.parametrize("forced", [True, False])
def test_even_nx_equals_packed_bitwise(size, kw, forced):
    fields = workloads.random_smooth(*size, seed=sum(size), vmax=0.05)
    forcing = FORCING if forced else None
    ref = _run("packed", *size, fields, forcing, **kw)
    if kw.get("cfl", 1.0) > 1.0:  # one node a thread: the same arithmetic up to the compiler's contractions
        got = _run("gather", *size, fields, forcing, **kw)
        assert np.max(np.abs(got - ref)) <= 1e-6 * np.max(np.abs(ref))
        return
    for block in (None, (32, 4), (256, 1)):
        np.testing.assert_array_equal(_run("gather", *size, fields, forcing, block, **kw), ref)


@pytest.mark.parametrize("size", [(5, 7), (33, 20), (131, 65)])
def test_odd_nx_matches_oracle(size):
    nx, ny = size
    fields = workloads.random_smooth(nx, ny, seed=nx, vmax=0.05)
    got = _run("gather", nx, ny, fields, FORCING)
    f = oracle.init(nx, ny, *fields)
    oracle.run(f, 0.6, 13, kmin=1, kmax=1, amp=1e-4, seed=3, redraw=7)
    # 13 steps of FP32 roundings of deviations of a few hundredths of W: the parity tests' 1e-5 of eps over 100 steps
    assert np.max(np.abs(got - oracle.merge_classes(f))) <= 1e-6 * np.max(np.abs(got))
