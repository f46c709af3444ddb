"""Handle-free batched Query and Recover (32-row panels whose warps split K) equal the oracle bit for
bit at the edges of a panel, of a slab of 128 columns and of the copy widths."""
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


def _dev_u32(a, offset=0):
    """The words on the device, `offset` words past an allocation's start."""
    buf = torch.zeros(a.size + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = pir.from_u32(np.ascontiguousarray(a, dtype=np.uint32).reshape(-1))
    return buf[offset:]


# (rows of A and H, n, B): panels of 4, 8, 16, 24 and 32 vectors, one and several per row block;
# rows and n just off 32 and 128; n a multiple of 4, of 2 and odd
SHAPES = [(1, 1, 2), (31, 3, 4), (32, 4, 5), (33, 127, 8), (70, 128, 9), (64, 129, 16), (100, 130, 17),
          (97, 256, 24), (130, 630, 25), (257, 384, 32), (65, 513, 33), (40, 1022, 70), (33, 2048, 130)]


@pytest.mark.parametrize("rows,n,B", SHAPES)
@pytest.mark.parametrize("offset", [0, 1, 2])   # words off 16-byte alignment: narrower copies
def test_query_and_recover(rows, n, B, offset):
    seed = 5 * rows + n + B
    A = inputs.uniform_u32(rows * n, seed=seed, tag=inputs.TAG_MISC).reshape(rows, n)
    S = inputs.secrets(B, n, seed=seed + 1)
    E = inputs.noise_batch(B, rows, seed=seed + 2)
    ans = inputs.uniform_u32(B * rows, seed=seed + 3, tag=inputs.TAG_MISC).reshape(B, rows)
    cols = inputs.target_columns(B, rows, seed=seed + 4)
    prm = pir.params(rows, rows, n, seed=seed)
    A_d, S_d = _dev_u32(A, offset), _dev_u32(S, offset)
    Q = torch.empty(B * rows, dtype=torch.int32, device="cuda")
    out = torch.empty(B * rows, dtype=torch.uint8, device="cuda")
    pir.qpadl_pir_query_batch(prm, A_d, S_d, torch.from_numpy(np.ascontiguousarray(E).reshape(-1)).cuda(),
                              torch.from_numpy(cols.astype(np.int32)).cuda(), Q)
    pir.qpadl_pir_recover_batch(prm, _dev_u32(ans), A_d, S_d, out)
    torch.cuda.synchronize()
    Q_np, out_np = pir.as_u32(Q).reshape(B, rows), out.cpu().numpy().reshape(B, rows)
    for b in range(B):
        assert np.array_equal(Q_np[b], oracle.query(A, S[b], E[b], int(cols[b]), 1 << 24)), b
        assert np.array_equal(out_np[b], oracle.recover(ans[b], A, S[b])), b


# products large enough for 128 x 128 tiles, rows of one- and two-word copies: whole tiles and ragged ones
@pytest.mark.parametrize("rows,n,B", [(8000, 33, 1024), (12801, 7, 1100), (20001, 34, 900), (9000, 101, 1025)])
def test_many_vectors(rows, n, B):
    seed = rows + n + B
    A = inputs.uniform_u32(rows * n, seed=seed, tag=inputs.TAG_MISC).reshape(rows, n)
    S = inputs.secrets(B, n, seed=seed + 1)
    E = inputs.noise_batch(B, rows, seed=seed + 2)
    ans = inputs.uniform_u32(B * rows, seed=seed + 3, tag=inputs.TAG_MISC).reshape(B, rows)
    cols = inputs.target_columns(B, rows, seed=seed + 4)
    prm = pir.params(rows, rows, n, seed=seed)
    A_d, S_d = _dev_u32(A), _dev_u32(S)
    Q = torch.empty(B * rows, dtype=torch.int32, device="cuda")
    out = torch.empty(B * rows, dtype=torch.uint8, device="cuda")
    pir.qpadl_pir_query_batch(prm, A_d, S_d, torch.from_numpy(np.ascontiguousarray(E).reshape(-1)).cuda(),
                              torch.from_numpy(cols.astype(np.int32)).cuda(), Q)
    pir.qpadl_pir_recover_batch(prm, _dev_u32(ans), A_d, S_d, out)
    torch.cuda.synchronize()
    Q_np, out_np = pir.as_u32(Q).reshape(B, rows), out.cpu().numpy().reshape(B, rows)
    for b in (0, 1, 31, 127, 128, 129, 511, B - 2, B - 1):
        assert np.array_equal(Q_np[b], oracle.query(A, S[b], E[b], int(cols[b]), 1 << 24)), b
        assert np.array_equal(out_np[b], oracle.recover(ans[b], A, S[b])), b
