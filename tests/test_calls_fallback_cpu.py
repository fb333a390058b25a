"""The binding without the extension over torch tensors: it imports, and the forward calls go through ctypes."""
import subprocess
import sys

import pytest

from paper_1606_00094_b200 import binding as B

MISSING = """
import os, warnings
from paper_1606_00094_b200 import build
build.calls_path = lambda: {path!r}
from paper_1606_00094_b200 import binding as B
assert B.boda_conv_out_dim(27, 5, 1, 2) == 27
with warnings.catch_warnings(record=True) as seen:
    warnings.simplefilter("always")
    calls = B._load_calls()
    assert B._load_calls() is calls
assert [w.category for w in seen] == [RuntimeWarning]
assert calls.planned(1, None, (1, 1, 1, 1), None, None, None, None) is None and calls.conv_fwd(1, 2, 3, 4, 5, 6) is None and calls.sgemm(1, 2, 3, 4, 5, 6) is None
try:
    B.boda_sgemm(None, None, None, 1, 1, 1, stream=0)
except B.BodaError as e:
    assert e.status == B.BODA_ERR_INVALID_ARG
else:
    raise AssertionError("no error")
"""


@pytest.mark.parametrize("kind", ["absent", "broken"])
def test_without_the_extension(kind, tmp_path):
    path = tmp_path / "_torch_calls.so"
    if kind == "broken":
        path.write_bytes(b"not a library")
    run = subprocess.run([sys.executable, "-c", MISSING.format(path=str(path))], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr


def test_with_the_extension():
    assert B._load_calls() is not B._CtypesOnly
