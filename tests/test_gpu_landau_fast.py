"""The Landau frame of the fused step (landau_fast) against the Newton solve
it stands in for, both measured against a long-double solve."""
import json
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(HERE, "numerics", "landau_fast_check.cu")


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("landau") / "check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-o", exe, SRC], check=True)
    return lambda *a: json.loads(subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                                text=True).stdout)


# |v| up to vmax: inside the FP32 early exit, across its edge (0.055) and far
# beyond it; then references and momenta FP32 cannot carry (FP64 only).  Both
# solves end with the same few roundings, so over 32768 states the mean error
# may differ by a quarter and the largest by a factor of two, or by two units
# in the last place where the solve's own error is smaller than that.
@pytest.mark.parametrize("vmax,eps0,tiny,fp32", [(0.01, 1.0, 1.0, True), (0.06, 1.0, 1.0, True),
                                                 (0.12, 3.0, 1.0, True), (0.6, 0.5, 1.0, True),
                                                 (0.95, 1.0, 1.0, True), (0.05, 1.0, 1e-14, False),
                                                 (0.05, 1.0, 1e-40, False), (0.3, 1e30, 1.0, False),
                                                 (0.3, 1e-30, 1.0, False)])
def test_landau_fast_is_as_accurate_as_the_newton_solve(check, vmax, eps0, tiny, fp32):
    r = check(vmax, eps0, tiny)
    assert r["widen_bad"] == 0, r  # FP32 -> FP64 on the integer pipe is the conversion, bit for bit
    for bits, unit in ((64, 2.0 ** -52), (32, 2.0 ** -23))[:2 if fp32 else 1]:
        assert r["fast%d_max" % bits] <= max(2.0 * r["solve%d_max" % bits], 2 * unit), r
        assert r["fast%d_mean" % bits] <= max(1.25 * r["solve%d_mean" % bits], unit), r
