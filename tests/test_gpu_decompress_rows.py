"""The row decompress kernel (planes of 2048 elements and more, or too large for the flat kernel's table; any width and block):
exact parity with the CPU checker where quads straddle rows, bands and planes, and at the smallest width it takes."""
import numpy as np
import pytest
import torch

from oracle import division_oracle as orc
from paper_2208_04187_b200 import binding, build, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built_library():
    build.build()
    binding.lib()


CASES = [   # n, c, h, w, block, q, x, lfc
    (2, 4, 75, 75, 8, 2, "f32", "bf16"), (2, 4, 5, 603, 16, 4, "f32", "f32"), (3, 4, 603, 5, 8, 8, "f32", "f32"),
    (2, 8, 47, 61, 12, 2, "bf16", "bf16"), (2, 2, 70, 90, 64, 1, "f32", "f32"), (1, 16, 46, 46, 4, 4, "bf16", "f32"),
    (2, 12, 2101, 7, 3, 2, "f32", "f32"), (1, 4, 517, 6, 1, 8, "f32", "f32"), (5, 3, 64, 33, 16, 2, "f32", "f32"),
]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_row_kernel_matches_the_checker(case):
    n, c, h, w, block, q, xd, ld = case
    x = synth.activation_map(n, c, h, w, "bn", 21 + w)
    x = synth.to_bf16_bits(x) if xd == "bf16" else x
    ref = orc.compress(x, block, q, 3, xd, ld)
    codec = binding.Codec(n, c, h, w, block, q, xd, ld)
    assert codec.plan().decompress_fast == 4
    codec.blob.copy_(torch.from_numpy(ref.blob()))
    pad = 1024
    out = torch.full((n * c * h * w + 2 * pad,), 7.0, dtype=binding.torch_dtype(xd), device="cuda")
    codec.decompress(out=out[pad:-pad].view(n, c, h, w))
    torch.cuda.synchronize()
    assert bool((out[:pad] == 7.0).all()) and bool((out[-pad:] == 7.0).all())
    got = out[pad:-pad]
    got = orc.bf16_bits_to_f32(got.view(torch.int16).cpu().numpy().view(np.uint16)) if xd == "bf16" else got.cpu().numpy()
    np.testing.assert_array_equal(got.reshape(n, c, h, w), orc.decompress(ref))
