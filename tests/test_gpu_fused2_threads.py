"""The 64 x 8 tiles of the FP32 two-step kernel at the edges of the rule that
picks the block's threads (up to 152 tiles, up to 304, more): bit for bit
against the packed single steps."""
import numpy as np
import pytest

import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402


# 152 tiles exactly and ragged, 153, 304, 304 ragged, 306
@pytest.mark.parametrize("size", [(1216, 64), (1154, 57), (576, 136), (1216, 128), (1156, 121), (1088, 144)])
@pytest.mark.parametrize("kw", [{}, dict(cfl=0.625)])
@pytest.mark.parametrize("forced", [True, False])
def test_equals_packed_single_steps(size, kw, forced):
    fields = workloads.random_smooth(*size, seed=size[1], vmax=0.05)
    out = []
    for kernel in ("packed", "fused2"):
        lat = rl.Lattice(*size, 0.6, dtype="f32", kernel=kernel, **kw,
                         forcing=dict(kmin=1, kmax=2, amp=1e-4, seed=3, redraw_period=7) if forced else None)
        if kernel == "fused2":
            lat.set_launch(kernel, 64, 8, 4)
        lat.init_fields(*fields)
        for n in (2, 5, 6):
            lat.step(n)
        out.append(lat.populations())
        lat.close()
    np.testing.assert_array_equal(out[1], out[0])
