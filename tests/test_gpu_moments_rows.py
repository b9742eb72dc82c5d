"""The moments kernel takes several nodes of a column per thread where the
lattice has blocks to spare: sides that leave a block's last rows and columns
ragged, at each number of rows, against the oracle."""
import os

import numpy as np
import pytest

import oracle
import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

oracle.set_threads(os.cpu_count() or 4)


# blocks of 32 columns and 8 r rows, r the largest of 8, 4, 2, 1 that leaves 608 of them: r = 1 (the last size below 2),
# 2, 4 and 8, with ny one past a block, one short of one and odd, nx one past 32 columns and one short
@pytest.mark.parametrize("size,rows", [((1023, 287), 1), ((1025, 297), 2), ((1023, 769), 4), ((993, 1313), 8),
                                       ((2048, 641), 8)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_ragged_sizes_match_oracle(size, rows, dtype):
    nx, ny = size
    blocks = {r: -(-nx // 32) * -(-ny // (8 * r)) for r in (8, 4, 2)}
    assert rows == next((r for r in (8, 4, 2) if blocks[r] >= 608), 1)
    fields = workloads.random_smooth(nx, ny, seed=nx + ny, deps=0.05, vmax=0.3)
    lat = rl.Lattice(nx, ny, 0.7, dtype=dtype)
    lat.init_fields(*fields)
    e, vx, vy, tot = lat.moments()
    lat.close()
    f = oracle.init(nx, ny, *fields)
    E, VX, VY = oracle.fields(f)
    # T^{0 mu} is linear in the populations; summed pairwise (the oracle's own totals add up node by node)
    want = oracle.moments(np.array([np.sum(fi) for fi in f]))[0, :3]
    # populations rounded once to the storage, moments of 17 of them: a few units in the last place of eps
    unit = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    assert np.max(np.abs(e - E)) <= 32 * unit * np.max(E)
    assert max(np.max(np.abs(vx - VX)), np.max(np.abs(vy - VY))) <= 32 * unit
    # the sums of nx ny such values: their errors add up to no more than that of a value times their number
    assert np.max(np.abs(np.asarray(tot)[:3] - want)) <= 32 * unit * nx * ny
