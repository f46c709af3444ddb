"""The largest exact sums of the four-limb Response: its chunks are up to 1024 deep, and centred digits of -128 times
byte limbs of -128 add up to 2^24 in a chunk.  Odd numbers of 64-query halves on a few thousand rows, where
four limbs are the faster form; sampled rows against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_03631_gb300 import inputs, pir

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,C,B", [(2304, 33001, 150), (3000, 32768, 140), (8192, 8200, 150)])
def test_largest_sums(R, C, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    D = inputs.db_digits(R, C, 256, seed=R)
    D[0::3] = 0      # -128 once centred
    D[1::3] = 255    # 127
    Q = inputs.uniform_u32(B * C, seed=B, tag=inputs.TAG_MISC).reshape(B, C)
    for b, word in enumerate((0x7F7F7F80, 0x7F7F7F7F, 0x80808080, 0xFFFFFFFF)):   # byte limbs -128, 127, -128.., -1
        Q[b::20] = word
    db = pir.qpadl_pir_setup(pir.params(R, C, 64), torch.from_numpy(D).cuda())
    out = torch.empty(B * R, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_answer_batch(db, pir.from_u32(Q.reshape(-1)), out)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    rows = np.array([0, 1, 2, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, R - 3, R - 2, R - 1])
    exp = oracle.answer_batch(np.ascontiguousarray(D[rows]), Q, threads=oracle.max_threads())
    assert np.array_equal(pir.as_u32(out).reshape(B, R)[:, rows], exp)
    db.close()
