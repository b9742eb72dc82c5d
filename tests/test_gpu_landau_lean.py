"""The FP32 frame does not lean to one side: rounding errors of single frames
average out over a flow, a lean adds up step by step in its totals."""
import json
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("lean") / "check")
    subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-o", exe, os.path.join(HERE, "numerics", "landau_lanes_check.cu")],
                   check=True)
    return lambda *a: json.loads(subprocess.run([exe, *map(str, a)], check=True, capture_output=True,
                                                text=True).stdout)


# A frame is rounded by about a unit, 2^-24, either way: over 32768 states that leaves 2^-24 / 181.  The early exit may
# leave a tenth of a unit, the sums of delta less than that.
@pytest.mark.parametrize("lo,hi", [(0.01, 0.03), (0.03, 0.043), (0.043, 0.05), (0.045, 0.055), (0.055, 0.07),
                                   (0.1, 0.2), (0.2, 0.5)])
def test_frames_average_to_the_solution(check, lo, hi):
    r = check(lo, hi)
    assert abs(r["lean_v"]) <= 2.0 ** -24 / 10, r
    assert abs(r["lean_delta"]) <= 2.0 ** -24 / 10, r
