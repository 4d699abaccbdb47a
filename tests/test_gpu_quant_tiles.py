"""The division-free quantiser: its premise checked by enumeration on the host, and its records compared with the
oracle's byte for byte at block sizes, alignments and values where a lane group or a threshold could go wrong."""
import numpy as np
import pytest
import torch

from gpu_util import as_f64
from oracle import quant
from paper_2503_15798_b200 import binding as mole

DEV = "cuda"
FMT = {4: mole.LUT_NF4, 3: mole.LUT_NF3}


@pytest.mark.parametrize("nbits,scale_bits", [(4, 8), (3, 11)])
def test_rounded_quotient_and_exact_product_agree_on_every_midpoint(nbits, scale_bits):
    """fl32(x / s) > m exactly when x > s m, for every mantissa of a bf16 x and of a scale of scale_bits bits."""
    cb = quant.nf_codebook_f32(nbits)
    mid = (np.float32(0.5) * (cb[:-1] + cb[1:])).astype(np.float32)
    x = np.arange(128, 256, dtype=np.float64)
    s = np.arange(2 ** (scale_bits - 1), 2 ** scale_bits, dtype=np.float64)
    for m in mid:
        for e in range(-8, 9):
            X, S = np.sign(float(m)) * (x * 2.0 ** (scale_bits - 8 + e))[:, None], s[None, :]
            y = X.astype(np.float32) / S.astype(np.float32)
            assert np.array_equal(y > m, X > S * float(m))  # s m: at most 35 bits, exact in float64


@pytest.mark.gpu
@pytest.mark.parametrize("nbits", [4, 3])
@pytest.mark.parametrize("N,d,block,V", [(4, 32, 32, 3), (3, 96, 96, 5), (5, 160, 160, 7), (4, 256, 64, 2), (16, 768, 768, 4), (2, 1152, 1152, 3),
                                         (1, 2048, 2048, 2), (1, 2048, 1024, 33), (1, 4096, 4096, 2), (7, 640, 128, 9)])
@pytest.mark.parametrize("offset", [0, 8])  # elements: a table that is 16- but not 32-byte aligned
def test_records_equal_the_oracles(nbits, N, d, block, V, offset):
    g = torch.Generator().manual_seed(N * d + V)
    lut = torch.empty(V, N, d).normal_(0, 0.05, generator=g).to(torch.bfloat16)
    lut[0, 0, :block] = 0.0                                    # scale zero
    lut[V - 1, N - 1, d - block:] *= 2.0 ** -110               # scales that underflow (float16) or take the dividing path
    lut[V // 2, 0, :block] = (torch.arange(block) % 251 - 125).to(torch.bfloat16)  # quotients on a fixed grid, both signs
    lut[V - 1, 0, 0] = 3.0e38                                  # above the largest float16 scale
    dev = torch.empty(lut.numel() + offset, dtype=torch.bfloat16, device=DEV)[offset:].view(V, N, d)
    dev.copy_(lut)
    want = quant.quantize_table(as_f64(lut).astype(np.float32), nbits, block)
    got = mole.QuantTable.quantize(dev, FMT[nbits], block).packed.cpu().numpy()
    assert np.array_equal(got, want)
