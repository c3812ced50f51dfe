"""The row-wise quantiser where its short division can go wrong: every row length it holds in registers and one that it does
not, quotients over the whole range of the format (its subnormals and the ties between codes too), zeros of both signs, rows
of zeros, scales outside the range of the short division and with an all-ones significand.  Codes and scales equal the
oracle's bit for bit."""
import numpy as np
import pytest
import torch

from oracle import fp8_oracle as f8
from paper_2107_05377_b200 import binding as mt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,cols", [(65, 256), (300, 768), (17, 1024), (300, 3072), (9, 4096)])
def test_codes_and_scales_equal_the_oracle(rows, cols):
    rng = np.random.default_rng(cols)
    x = rng.standard_normal((rows, cols)) * np.exp2(rng.integers(-22, 1, (rows, cols)))
    x *= np.exp2(rng.integers(-90, 90, (rows, 1)).astype(np.float64))     # scales inside and outside 2^-60 .. 2^60
    x[1::8] = np.exp2(rng.integers(-14, 9, x[1::8].shape)) * rng.integers(8, 32, x[1::8].shape)   # few significant bits:
    x[1::8, 0] = 448.0 * 32.0                                             # scale 32 exactly, quotients on the ties
    x[2::8, ::3] = 0.0
    x[3::8, ::3] = -0.0
    x[4] = 0.0
    xt = torch.from_numpy(x).to(torch.bfloat16)
    # an all-ones significand of amax / 448: the bf16 values of one binade that give it, if any, as the largest of a row
    cand = torch.arange(0x3F80, 0x4000, dtype=torch.int32).to(torch.int16).view(torch.bfloat16)
    scale = (cand.float() * np.float32(1.0 / 448.0)).view(torch.int32) & 0x7FFFFF
    near = int(torch.argmax(scale))
    xt[5] = (torch.rand(cols) * 0.9).to(torch.bfloat16)
    xt[5, 0] = cand[near]
    q = torch.zeros(rows, cols, dtype=torch.uint8, device="cuda")
    s = torch.zeros(rows, device="cuda")
    mt.mt_kernel_quantize_rows(xt.cuda(), q, s)
    torch.cuda.synchronize()
    want_q, want_s = f8.quantize_rows(xt.float().numpy().astype(np.float64))
    assert np.array_equal(s.cpu().numpy(), want_s)
    assert np.array_equal(q.cpu().numpy(), want_q)
