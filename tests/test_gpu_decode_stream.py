"""GPU parity of hif8_decode to 16-bit formats where the kernel with a table per lane takes over (2^21 codes) and at the ends of its
blocks and vectors, bit for bit: the 256 values come from the oracle, every result is one of them."""
import numpy as np
import pytest
import torch

import paper_2409_16626_b200 as H
from oracle import hif8_oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,scale_exp", [(H.BF16, 0), (H.BF16, 120), (H.F16, 3), (H.F16, -20)])
@pytest.mark.parametrize("n", [(1 << 21) - 1, 1 << 21, (1 << 21) + 7, 130 * 16384, 130 * 16384 + 16383, 3001 * 4099])
@pytest.mark.parametrize("src_off,dst_off", [(0, 0), (8, 16), (3, 0), (0, 2)])
def test_decode_large_16_bit(n, dtype, scale_exp, src_off, dst_off):
    codes = np.random.default_rng(n + src_off).integers(0, 256, n, dtype=np.uint8)
    table = O.decode(np.arange(256, dtype=np.uint8), dtype, scale_exp)
    src = torch.empty(n + src_off, dtype=torch.uint8, device="cuda")
    src[src_off:].copy_(torch.from_numpy(codes))
    dst = torch.full((2 * n + dst_off + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    H.hif8_decode(src.data_ptr() + src_off, dst.data_ptr() + dst_off, dtype, n, scale_exp)
    got = dst.cpu().numpy()
    assert np.all(got[:dst_off] == 0xA5) and np.all(got[dst_off + 2 * n:] == 0xA5)
    assert np.array_equal(got[dst_off:dst_off + 2 * n].copy().view(np.uint16), np.asarray(table).view(np.uint16)[codes])
