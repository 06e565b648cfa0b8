"""The 8-bit quantiser over its whole input range and at the edges of its grid, against the oracle.

Rows of arbitrary finite bf16 bit patterns (subnormals and both zeros among them) meet every
combination of exponents; the row counts leave partial blocks and partial warps.
"""
import numpy as np
import pytest
import torch

from oracle.q8 import quantise_rows
from paper_2511_22481_b200 import binding as B

pytestmark = pytest.mark.gpu


def _quantise(bits):
    rows = torch.from_numpy(bits.view(np.int16)).view(torch.bfloat16).cuda()
    n = rows.shape[0]
    codes = torch.full((n + 1, B.OMNI_Q8_ROW_BYTES), 0xA5, dtype=torch.uint8, device="cuda")
    scale = torch.full((n + 1,), -1.0, device="cuda")
    B.omni_kv_quantize_q8(rows, codes[:n], scale[:n])
    torch.cuda.synchronize()
    assert bool((codes[n] == 0xA5).all()) and float(scale[n]) == -1.0      # nothing past the last row
    return codes[:n].cpu().numpy(), scale[:n].cpu().numpy()


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 33, 4001])
def test_any_finite_bits(n):
    rng = np.random.default_rng(n)
    # a window of exponents per row, so that codes of every size occur, and all exponents at once
    low = rng.integers(0, 255, size=(n, 1))
    width = rng.choice([1, 4, 12, 255], size=(n, 1))
    exponent = np.minimum(low + rng.integers(0, 255, size=(n, 576)) % width, 254)
    bits = (rng.integers(0, 2, size=(n, 576)) << 15 | exponent << 7 | rng.integers(0, 128, size=(n, 576))).astype(np.uint16)
    bits[:, 7::97] = 0x8000                                                # -0 keeps its sign
    if n > 2:
        bits[1, :512] = 0x8000
    codes, scale = _quantise(bits)
    with np.errstate(all="ignore"):
        want_codes, want_scale = quantise_rows(bits)
    assert np.array_equal(scale.view(np.uint32), want_scale.view(np.uint32))
    assert np.array_equal(codes, want_codes)


def test_infinity_and_nan():
    """Division semantics: a row with an infinity has scale inf, its finite values become zeros of their
    sign and inf / inf is NaN; a NaN is coded as NaN and takes no part in the maximum."""
    bits = np.full((3, 576), 0x3F80, dtype=np.uint16)
    bits[0, 5], bits[0, 6], bits[0, 7] = 0x7F80, 0xFF80, 0xBF80
    bits[1, 300] = 0x7FC0
    codes, scale = _quantise(bits)
    assert np.isinf(scale[0]) and scale[1] == scale[2] == np.float32(1) / np.float32(448)
    assert codes[0, 0] == 0 and codes[0, 5] == codes[0, 6] == 0x7F and codes[0, 7] == 0x80
    assert codes[1, 300] == 0x7F
    keep = np.arange(640) != 300
    assert np.array_equal(codes[1][keep], codes[2][keep])
