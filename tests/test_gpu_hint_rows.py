"""Row-major outputs of the hint on pair tiles: rows of 16-byte stores, and rows whose length or place does not allow
them, which are turned over the lanes of a warp; whole tiles and column ranges that add up."""
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


# one word short of and past groups of 32, 64, 128 and 192 vectors; rows short of and past 32 and 256
@pytest.mark.parametrize("n", [66, 95, 96, 127, 129, 191, 193, 260])
@pytest.mark.parametrize("R,C", [(1, 300), (31, 129), (33, 700), (257, 512), (300, 9000), (1100, 1300)])
@pytest.mark.parametrize("shift", [0, 1])   # the hint on and off a 16-byte boundary
def test_hint_rows(R, C, n, shift):
    D, A = inputs.db_digits(R, C, 256, seed=R), inputs.public_matrix(C, n, seed=n)
    db = pir.qpadl_pir_setup(pir.params(R, C, n), torch.from_numpy(D).cuda())
    buf = torch.full((R * n + 8,), -1, dtype=torch.int32, device="cuda")
    H = buf[shift:shift + R * n]
    pir.qpadl_pir_hint(db, pir.from_u32(A.reshape(-1)), H)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    assert np.array_equal(pir.as_u32(H).reshape(R, n), oracle.hint(D, A, threads=oracle.max_threads()))
    assert (buf[:shift] == -1).all() and (buf[shift + R * n:] == -1).all()
    db.close()
