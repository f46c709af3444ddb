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


# blocks staged whole (up to 80 entries) and the first tiled length; 1, 127 to 132 and many columns; the ragged last
# block; rows of whole words and not
@pytest.mark.parametrize("E", [1, 2, 3, 5, 16, 64, 79, 80, 81])
@pytest.mark.parametrize("C,short", [(1, 0), (3, 1), (127, 0), (128, 1), (132, 2), (2000, 0)])
@pytest.mark.parametrize("w", [1, 2, 3, 4])
def test_encode_of_short_blocks(E, C, short, w):
    n = max(1, C * E - short)
    C = -(-n // E)
    x = inputs.uniform_u32(n, seed=n + w, tag=inputs.TAG_MISC)   # the encoder keeps w bytes of any difference
    for at in (0, 1):   # the database on and off a 4-byte boundary
        buf = torch.full((pir.delta_rows(E, w) * C + at,), 0xAB, dtype=torch.uint8, device="cuda")
        pir.qpadl_pir_delta_encode(torch.from_numpy(x.view(np.int32)).cuda(), E, w, buf[at:])
        got = buf[at:].cpu().numpy().reshape(-1, C)
        v = np.concatenate([x, np.full(C * E - n, x[-1], dtype=np.uint32)]).reshape(C, E)
        d = v[:, 1:] - v[:, :-1]
        exp = [(v[:, 0] >> np.uint32(8 * k)) & 255 for k in range(4)]
        exp += [(d[:, i] >> np.uint32(8 * k)) & 255 for i in range(E - 1) for k in range(w)]
        assert np.array_equal(got, np.array(exp, dtype=np.uint8))
        assert at == 0 or int(buf[0]) == 0xAB


# CTAs of one warp, of two, of 31 and of 32, one run and two; many blocks
@pytest.mark.parametrize("E", [1, 2, 255, 256, 257, 512, 513, 7936, 7937, 8192, 8193])
@pytest.mark.parametrize("w,B", [(1, 1), (2, 70), (4, 5)])
def test_decode_warps_per_block(E, w, B):
    Rp = pir.delta_rows(E, w)
    digits = np.ascontiguousarray(inputs.uniform_u32((B * Rp + 3) // 4, seed=E + w, tag=inputs.TAG_MISC)
                                  .view(np.uint8)[:B * Rp]).reshape(B, Rp)
    out = torch.full((B * E + 8,), -1, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_delta_decode(torch.from_numpy(digits).cuda(), B, E, w, out[:B * E])
    got = pir.as_u32(out)
    exp = np.stack([oracle.delta_decode(digits[b], E, w) for b in range(B)])
    assert np.array_equal(got[:B * E].reshape(B, E), exp)
    assert (got[B * E:] == 0xFFFFFFFF).all()


# few long blocks, written as one run of bytes: the first column counts past the line too, ragged last blocks, the database
# on and off a 4-byte boundary
@pytest.mark.parametrize("C", [1, 2, 3, 5, 16, 28, 29, 32, 33, 40, 41])
@pytest.mark.parametrize("E,short", [(81, 0), (82, 80), (1001, 3), (4097, 4000)])
@pytest.mark.parametrize("w", [1, 2, 3, 4])
def test_encode_of_few_blocks(C, E, short, w):
    n = C * E - short
    C = -(-n // E)
    x = inputs.uniform_u32(n, seed=n + w, tag=inputs.TAG_MISC)
    for at in (0, 1):
        buf = torch.full((pir.delta_rows(E, w) * C + at + 5,), 0xAB, dtype=torch.uint8, device="cuda")
        end = buf.numel() - 5
        pir.qpadl_pir_delta_encode(torch.from_numpy(x.view(np.int32)).cuda(), E, w, buf[at:end])
        v = np.concatenate([x, np.full(C * E - n, x[-1], dtype=np.uint32)]).reshape(C, E)
        d = v[:, 1:] - v[:, :-1]
        exp = np.empty((4 + (E - 1) * w, C), dtype=np.uint8)
        for k in range(4):
            exp[k] = (v[:, 0] >> np.uint32(8 * k)) & 255
        for k in range(w):
            exp[4 + k::w] = ((d >> np.uint32(8 * k)) & 255).T
        assert np.array_equal(buf[at:end].cpu().numpy().reshape(-1, C), exp)
        assert (buf[end:] == 0xAB).all() and (at == 0 or int(buf[0]) == 0xAB)
