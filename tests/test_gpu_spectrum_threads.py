"""Spectra of several handles from several host threads: one handle's shared
memory is not limited by another's smaller transform."""
import json
import os
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2101_06187_gb300 as rl  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    rl.library()  # built
    exe, lib = str(tmp_path_factory.mktemp("threads") / "check"), os.path.dirname(os.path.abspath(rl.__file__))
    subprocess.run(["g++", "-O2", "-std=c++17", "-pthread", "-o", exe,
                    os.path.join(HERE, "numerics", "spectrum_threads_check.cpp"), "-L" + lib, "-l:librlbm.so",
                    "-Wl,-rpath," + lib], check=True)
    return lambda *a: json.loads(subprocess.run([exe, *map(str, a)], check=True, capture_output=True, text=True,
                                                timeout=60).stdout)


# lines of 8192 points against shorter ones, in the row and in the column kernel; shells add to a line's memory
@pytest.mark.parametrize("long,short,nlong,nshort,along_y", [(8192, 4096, 8, 8, 0), (8192, 4096, 4096, 16, 1)])
def test_threads_take_spectra(check, long, short, nlong, nshort, along_y):
    r = check(long, short, nlong, nshort, along_y)
    assert r["error"] == "" and r["long"] > 0 and r["short"] > 0, r
