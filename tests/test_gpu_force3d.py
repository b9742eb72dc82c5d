"""The 3D stirring force summed by runs and groups of modes, at the edges of
its tiles (16 layers a thread, 32 x 8 columns a block), against the oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402


# fewer layers than one thread takes, exactly one, one more, several; ragged columns; one group (kz = 0 and 1 only)
@pytest.mark.parametrize("size,kmin,kmax", [((10, 9, 9), 1, 1), ((33, 15, 16), 1, 4), ((30, 17, 17), 2, 3),
                                            ((64, 24, 35), 4, 6), ((31, 40, 12), 1, 5)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_force_matches_oracle(size, kmin, kmax, dtype):
    nx, ny, nz = size
    amp, seed = 1e-3, 77
    lat = rl.Lattice3D(nx, ny, nz, 0.7, dtype=dtype,
                       forcing=dict(kmin=kmin, kmax=kmax, amp=amp, seed=seed, redraw_period=2))
    # every mode contributes at most 2 amp, off by a few units in the last place in its tables and products
    nmodes = lat.info()["nmodes"]
    tol = 8 * (2.0 ** -53 if dtype == "f64" else 2.0 ** -24) * 2 * amp * nmodes
    for epoch in range(2):
        ref = oracle.lattice3d.force_field(nx, ny, nz, kmin, kmax, amp, seed, epoch)
        for got, want in zip(lat.force(), ref):
            assert np.max(np.abs(got - np.asarray(want).reshape(got.shape))) <= tol
        lat.step(2)
    lat.close()
