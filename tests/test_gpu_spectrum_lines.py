"""The line transform of the spectra at lengths that take each of its passes
(radices 8, 4, 2, 3, 5, 7, larger primes, the longest lines), with all modes
wanted and with few of them, against numpy's FFT of the same velocity."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

# each axis of a size is a line length: powers of two (one pass to five), 3, 5 and 7 alone and mixed, primes above 7
# (first and later passes, the longest), lengths above 2048 (one line a block)
SIZES = [(4, 8), (6, 5), (7, 9), (11, 13), (64, 49), (96, 125), (121, 250), (127, 48), (512, 33), (384, 16),
         (1021, 6), (2048, 12), (22, 1009), (4095, 4), (8192, 4), (4, 8186), (8191, 4), (300, 320)]


@pytest.mark.parametrize("size", SIZES)
def test_spectrum_matches_numpy(size):
    nx, ny = size
    rng = np.random.default_rng(nx * 10000 + ny)
    lat = rl.Lattice(nx, ny, 0.8, dtype="f64")
    lat.init_fields(1.0 + 0.01 * rng.standard_normal((ny, nx)), 0.01 * rng.uniform(-1, 1, (ny, nx)),
                    0.01 * rng.uniform(-1, 1, (ny, nx)))
    _, vx, vy, _ = lat.moments()
    most = min(4096, int(np.hypot(nx / 2, ny / 2)) + 2)
    # a mode is a sum of nx ny values, each a few units off after log2(n) passes or a sum of n terms: 1e-13 of the
    # root-mean-square mode, which enters a shell's power linearly
    total = oracle.energy_spectrum(vx, vy, most).sum()
    for nshells in (1, 3, min(17, most), most):
        want = oracle.energy_spectrum(vx, vy, nshells)
        got = lat.energy_spectrum(nshells)
        assert np.all(np.abs(got - want) <= 1e-13 * np.sqrt(want * total) + 1e-13 * want + 1e-26 * total), nshells
    for kf in (0.0, 1.0, 2.5, 0.4 * min(nx, ny), 1e9):
        want = oracle.filtered_velocity_rms(vx, vy, kf)
        assert abs(lat.filtered_velocity(kf) - want) <= 1e-13 * np.sqrt(2 * total), kf
    lat.close()
