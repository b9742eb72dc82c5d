"""The two routes of the 3D stirring force: summed by runs and groups (FP64 and
FP32 storage), and mode by mode (16-bit storage, whose results stay those of
this order, and lattices without room for the sums)."""
import ctypes

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

SIZE, BAND, AMP, SEED = (33, 24, 19), (1, 4), 1e-3, 77
FORCING = dict(kmin=BAND[0], kmax=BAND[1], amp=AMP, seed=SEED, redraw_period=2)


class _Hooked(rl.Lattice3D):
    """A lattice whose ``refuse``-th allocation is refused (None: none is)."""

    def __init__(self, *a, refuse=None, **kw):
        self.refuse, self.calls, self.live = refuse, 0, {}
        super().__init__(*a, allocator="none", **kw)

    def _create(self, forcing, opts):
        def _alloc(nbytes, _ctx):
            self.calls += 1
            if self.calls - 1 == self.refuse:
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            self.live[t.data_ptr()] = t
            return t.data_ptr()

        def _free(ptr, _nbytes, _ctx):
            self.live.pop(int(ptr), None)

        self.hooks = rl.ALLOC_FN(_alloc), rl.FREE_FN(_free)
        opts.alloc, opts.free = self.hooks
        return super()._create(forcing, opts)


def _mode_by_mode(dtype):
    """A lattice whose optional last allocation, the sums' room, is refused."""
    probe = _Hooked(*SIZE, 0.7, dtype=dtype, forcing=FORCING)
    most = probe.calls
    probe.close()
    assert not probe.live
    return _Hooked(*SIZE, 0.7, dtype=dtype, forcing=FORCING, refuse=most - 1)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_refused_sums_leave_the_force_mode_by_mode(dtype):
    lat = _mode_by_mode(dtype)
    # every mode contributes at most 2 amp, off by a few units in the last place in its tables and products
    tol = 8 * (2.0 ** -53 if dtype == "f64" else 2.0 ** -24) * 2 * AMP * lat.info()["nmodes"]
    for epoch in range(2):
        ref = oracle.lattice3d.force_field(*SIZE, *BAND, AMP, SEED, epoch)
        for got, want in zip(lat.force(), ref):
            assert np.max(np.abs(got - np.asarray(want).reshape(got.shape))) <= tol
        lat.step(2)
    lat.synchronize()
    lat.close()
    assert not lat.live


# The 16-bit forms compute in FP32, so their force is FP32's mode by mode, bit for bit.
@pytest.mark.parametrize("dtype", ["bf16", "f16"])
def test_16bit_force_is_the_mode_by_mode_one(dtype):
    ref = _mode_by_mode("f32")
    lat = rl.Lattice3D(*SIZE, 0.7, dtype=dtype, forcing=FORCING)
    for epoch in range(2):
        for got, want in zip(lat.force(), ref.force()):
            np.testing.assert_array_equal(got, want)
        lat.step(2)
        ref.step(2)
    lat.close()
    ref.close()


def test_refused_needed_allocation_is_reported():
    """Any earlier allocation is needed: the create fails and frees what it got."""
    probe = _Hooked(*SIZE, 0.7, forcing=FORCING)
    most = probe.calls
    probe.close()
    for at in range(most - 1):
        live, calls = {}, [0]

        def _alloc(nbytes, _ctx):
            calls[0] += 1
            if calls[0] - 1 == at:
                return None
            t = torch.empty(int(nbytes), dtype=torch.uint8, device="cuda")
            live[t.data_ptr()] = t
            return t.data_ptr()

        def _free(ptr, _nbytes, _ctx):
            live.pop(int(ptr), None)

        hooks = rl.ALLOC_FN(_alloc), rl.FREE_FN(_free)
        o = rl.rlbm_opts_default()
        o.alloc, o.free = hooks
        out = ctypes.c_void_p()
        forcing = rl.Forcing(*BAND, AMP, SEED, 2)
        st = rl.library().rlbm_create3d(*SIZE, 0.7, ctypes.byref(forcing), ctypes.byref(o), ctypes.byref(out))
        assert st == rl.RLBM_ERR_ALLOC and out.value is None and not live, at
