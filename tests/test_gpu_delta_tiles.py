"""Compression kernels at the edges of their tiles (128 columns x 128 positions, runs of 8192 decoded
entries, 16-byte loads) equal the oracle's bytes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_03631_gb300 import inputs, pir

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)


# (entries, block, largest gap): one entry; blocks of 1, 127, 128, 129 and 8193 entries; 127..132
# blocks; ragged last blocks; widths 1 to 4
SHAPES = [(1, 1, 9), (4, 1, 9), (127 * 128, 128, 200), (128 * 128, 128, 300), (129 * 129 - 5, 129, 70000),
          (132 * 256, 256, 255), (131 * 127 + 1, 127, 2 ** 25), (3 * 8193, 8193, 31), (1 << 20, 8192, 31),
          (130 * 1000 - 1, 1000, 2000), (7, 300, 5)]


@pytest.mark.parametrize("n,E,gap", SHAPES)
@pytest.mark.parametrize("offset", [0, 1])   # entries off 16-byte alignment
def test_width_encode_decode(n, E, gap, offset):
    x = inputs.uniform_u32(n, seed=n + E, tag=inputs.TAG_MISC) % np.uint32(gap + 1)
    x = np.cumsum(x, dtype=np.uint32)
    buf = torch.zeros(n + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(x.view(np.int32)).cuda()
    xd = buf[offset:]
    w = pir.qpadl_pir_delta_width(xd, E)
    assert w == oracle.delta_width(x, E)
    C, Rp = (n + E - 1) // E, pir.delta_rows(E, w)
    db = torch.full((Rp * C,), 0xAB, dtype=torch.uint8, device="cuda")
    pir.qpadl_pir_delta_encode(xd, E, w, db)
    out = torch.empty(C * E + offset, dtype=torch.int32, device="cuda")[offset:]
    pir.qpadl_pir_delta_decode(db.view(Rp, C).t().contiguous(), C, E, w, out)
    torch.cuda.synchronize()
    assert np.array_equal(db.cpu().numpy().reshape(Rp, C), oracle.delta_encode(x, E, w))
    assert np.array_equal(pir.as_u32(out), np.concatenate([x, np.full(C * E - n, x[-1], dtype=np.uint32)]))


@pytest.mark.parametrize("at", [0, 1, 3, 511, 512, 513, 4095])
def test_width_sees_one_large_difference(at):
    # the only difference above one byte sits at `at`; one that crosses two blocks does not count
    x = np.arange(4096, dtype=np.uint32)
    x[at:] += 70000
    assert pir.qpadl_pir_delta_width(torch.from_numpy(x.view(np.int32)).cuda(), 512) == oracle.delta_width(x, 512)
