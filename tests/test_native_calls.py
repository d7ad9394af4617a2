"""The codec's calls through the CPython extension, as far as they need no GPU: tensors that cannot answer end in a
Python exception, and a codec is an ordinary object (it can be copied, sent to another process, given another descriptor)."""
import copy
import os
import pickle
import subprocess
import sys

import pytest
import torch
from torch.utils._python_dispatch import TorchDispatchMode

from paper_2208_04187_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()


# `without` has no storage to ask for; `x` stands for a CUDA tensor on a machine without one
STORAGELESS = """
import torch
from torch.utils._python_dispatch import TorchDispatchMode
from torch._subclasses.fake_tensor import FakeTensorMode
from paper_2208_04187_b200 import binding
without = torch.zeros(4096, dtype=torch.uint8).to_sparse()
with FakeTensorMode():
    x = torch.empty(2, 3, 8, 8, device="cuda")
desc = binding.make_desc(2, 3, 8, 8, 8, 2)
codec = object.__new__(binding.{cls})
codec.__dict__.update(desc=desc, blob=without, workspace=torch.zeros(4096, dtype=torch.uint8), device=torch.device("cpu"))
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


def codec_on_the_host(cls):
    """A codec whose buffers are on the host, through its own constructor: the library refuses its calls by the
    buffers' sizes, before any of them is touched."""
    return cls(2, 3, 8, 8, 8, 2, device="cpu")


@pytest.mark.parametrize("cls", [binding.Codec, binding.PlaneGroupCodec])
def test_codecs_can_be_copied_and_pickled(cls):
    codec = codec_on_the_host(cls)
    for twin in (copy.deepcopy(codec), pickle.loads(pickle.dumps(codec)), copy.copy(codec)):
        assert bytes(twin.desc) == bytes(codec.desc) and twin.shape == codec.shape and twin.blob.numel() == codec.blob.numel()
        assert not any(isinstance(v, type(os)) for v in vars(twin).values())


@pytest.mark.parametrize("cls", [binding.Codec, binding.PlaneGroupCodec])
def test_a_codec_follows_its_descriptor(cls, monkeypatch):
    """The call is made with the descriptor that the codec has now, not with one that it had when it was made."""
    codec = codec_on_the_host(cls)
    codec.blob = torch.zeros(16, dtype=torch.uint8)[:1]                # too small for either descriptor
    seen = []

    class Spy:
        def decompress(self, desc, *rest):
            seen.append(bytes(desc))
            return binding.DIV_ERR_CAPACITY
    monkeypatch.setattr(binding, "_native", Spy())
    for w in (8, 24):
        codec.desc = binding.make_desc(2, 3, 8, w, 8, 2)
        with pytest.raises(binding.DivisionError):
            codec.decompress()
        assert seen[-1] == bytes(codec.desc)


class Takes(Exception):
    pass


@pytest.mark.parametrize("cls", [binding.Codec, binding.PlaneGroupCodec])
def test_the_output_is_made_on_the_codec_s_device(cls):
    """Not on the blob's: a blob in pinned host memory, which the GPU reads in place, is rebuilt on the GPU."""
    codec = codec_on_the_host(cls)
    codec.device = torch.device("meta")
    made = []

    class Watch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            if func is torch.ops.aten.empty.memory_format:
                made.append((list(args[0]), kwargs.get("device"), kwargs.get("dtype")))
                raise Takes                     # before the call itself
            return func(*args, **(kwargs or {}))

    with Watch(), pytest.raises(Takes):
        codec.decompress()
    assert made == [([2, 3, 8, 8], torch.device("meta"), torch.float32)]


@pytest.mark.gpu
@pytest.mark.parametrize("cls", [binding.Codec, binding.PlaneGroupCodec])
def test_a_blob_in_pinned_host_memory_is_rebuilt_on_the_gpu(cls):
    x = torch.randn(2, 16, 28, 28, device="cuda")
    codec = cls(2, 16, 28, 28, 8, 2)
    codec.compress(x, seed=3)
    want = codec.decompress()
    host = codec.blob.cpu().pin_memory()
    got = codec.decompress(blob=host)
    assert got.device == want.device and torch.equal(got, want)
