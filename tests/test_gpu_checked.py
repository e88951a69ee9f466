"""The checked build (libamgd_checked.so, compiled with AMGD_CHECKS): every
gather index the sweep and distance kernels read from the matrix -- a column
index, a renumbered column or a row map -- is tested against the vector block
inside the kernel before its load.

* The GPU parity tests, run in a child process against the checked build,
  pass unchanged: on every shape, stage and storage they exercise no index
  fails its test, and the results are the normal build's.
* A column index planted out of range after the handle's setup is caught by
  the sweep's test and reported as AMGD_ERR_CHECK by the next synchronising
  call; the load itself is redirected to row 0 and never leaves the buffer.
* The entries of the sliced copy that a sweep asks the L2 for ahead of use are
  tested in the same way: none lies past the copy's end.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checked_lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1106_5990_gb300 import _build
    _build.build()
    return _build.build(checked=True)


def _child(args, **env_extra):
    env = dict(os.environ, AMGD_CHECKED="1", **env_extra)
    return subprocess.run([sys.executable, *args], cwd=ROOT, env=env, capture_output=True,
                          text=True, timeout=1800)


def test_child_loads_the_checked_build(checked_lib):
    p = _child(["-c", "from paper_1106_5990_gb300 import amgd; print(amgd.amgd_checked_build())"])
    assert p.returncode == 0 and p.stdout.strip() == "1", p.stdout + p.stderr
    p = subprocess.run([sys.executable, "-c", "from paper_1106_5990_gb300 import amgd; "
                        "print(amgd.amgd_checked_build())"], cwd=ROOT, capture_output=True,
                       text=True, timeout=600,
                       env={k: v for k, v in os.environ.items() if k != "AMGD_CHECKED"})
    assert p.returncode == 0 and p.stdout.strip() == "0", p.stdout + p.stderr


def test_parity_tests_pass_under_the_checked_build(checked_lib):
    p = _child(["-m", "pytest", "-x", "-q", "-p", "no:cacheprovider",
                "tests/test_gpu_parity.py", "tests/test_gpu_mixed.py", "tests/test_gpu_depth.py"])
    assert p.returncode == 0, p.stdout[-4000:] + p.stderr[-4000:]


PLANTED = r'''
from paper_1106_5990_gb300 import amgd, inputs
assert amgd.amgd_checked_build() == 1
rp, col, val = inputs.poisson2d_5pt(40)                  # 1600 rows, slot 77 exists
with amgd.Handle(rp, col, val, 8, 1) as h:
    h.set_kernel_shape(amgd.AMGD_KERNEL_RELAX, 4, 1, 4, 0)   # the direct sweep kernel
    h.relax(1, 0.7)
    try:
        h.get_vectors()                                    # synchronises: reads the status
    except amgd.AmgdError as e:
        assert e.status == amgd.AMGD_ERR_CHECK, e
        print("caught")
    else:
        raise SystemExit("the planted column was not reported")
'''


def test_planted_column_is_caught(checked_lib):
    p = _child(["-c", PLANTED], AMGD_TEST_BAD_COLUMN="77")
    assert p.returncode == 0 and p.stdout.strip().endswith("caught"), p.stdout + p.stderr


# 16 rows of 64 bytes per group, three groups per warp, the last group in the upper
# half of the last slice; and the other row widths at the same row counts
AHEAD = r'''
import torch
from paper_1106_5990_gb300 import amgd, inputs
assert amgd.amgd_checked_build() == 1
for n in (111872, 111872 - 16, 111872 - 37):
    rp, col, val = inputs.lap1d(n)
    for K in (2, 4, 8, 16, 32, 64):
        for prec in ("fp64", "fp32"):
            with amgd.Handle(rp, col, val, K, 1) as h:
                h.set_precision(prec)
                h.graph_capture(1, 1, 0.7, 0, 0.5, torch.empty(n + 1, dtype=torch.int64, device="cuda"),
                                torch.empty(len(col), dtype=torch.int32, device="cuda"))
                h.relax(1, 0.7)                  # reads the sliced copy
                h.get_vectors()                  # synchronises: reads the status
print("in range")
'''


def test_entries_asked_for_ahead_stay_in_the_copy(checked_lib):
    p = _child(["-c", AHEAD])
    assert p.returncode == 0 and p.stdout.strip().endswith("in range"), p.stdout + p.stderr
