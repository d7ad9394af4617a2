"""The codec's calls through the CPython extension, as far as they need no GPU: tensors that cannot answer end in a
Python exception."""
import os
import subprocess
import sys

import pytest

from paper_2208_04187_b200 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()


# `without` has no storage to ask for; `x` stands for a CUDA tensor on a machine without one
STORAGELESS = """
import ctypes, torch
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2208_04187_b200 import binding
without = torch.zeros(4096, dtype=torch.uint8).to_sparse()
with FakeTensorMode():
    x = torch.empty(2, 3, 8, 8, device="cuda")
desc = binding.make_desc(2, 3, 8, 8, 8, 2)
codec = object.__new__(binding.{cls})
codec.__dict__.update(desc=desc, blob=without, workspace=torch.zeros(4096, dtype=torch.uint8), device=torch.device("cpu"),
                      _native=binding.native(), _addr=ctypes.addressof(desc))
for call in (lambda: codec.compress(x), codec.decompress, lambda: codec.decompress(out=without)):
    try:
        call()
    except RuntimeError as e:
        assert "data pointer" in str(e), e
        print("raised")
"""


@pytest.mark.parametrize("cls", ["Codec", "PlaneGroupCodec"])
def test_a_tensor_without_storage_is_an_exception(cls):
    got = subprocess.run([sys.executable, "-c", STORAGELESS.format(cls=cls)], cwd=ROOT, capture_output=True, text=True,
                         env=dict(os.environ, PYTHONPATH=ROOT), timeout=300)
    assert got.returncode == 0 and got.stdout.split() == ["raised"] * 3, (got.returncode, got.stderr[-2000:])
