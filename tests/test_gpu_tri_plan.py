"""Products of few tiles: many short column ranges, of as little as two chunks of 128 columns, over tiles of one, two and
three 64-vector halves; answers and hints equal the oracle's, and a second call finds the output the first one left."""
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


@pytest.mark.parametrize("R,C,B", [(1, 255, 65), (1, 256, 65), (5, 513, 66), (300, 512, 160), (257, 1025, 129), (300, 4000, 66),
                                   (300, 4001, 190), (200, 19001, 100), (1200, 1900, 250), (700, 2500, 321), (2600, 900, 320),
                                   (100, 9000, 600), (255, 12289, 64)])
@pytest.mark.parametrize("digit", [None, 255])
def test_few_tiles(R, C, B, digit):
    D = inputs.db_digits(R, C, 256, seed=R) if digit is None else np.full((R, C), digit, dtype=np.uint8)
    Q = inputs.uniform_u32(B * C, seed=C + B, tag=inputs.TAG_MISC).reshape(B, C)
    Q[0] = 0xFFBFFC00   # every limb at its lowest
    db = pir.qpadl_pir_setup(pir.params(R, C, B), torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_U8_MAX_BATCH, 0)
    out = torch.full((B * R,), -1, dtype=torch.int32, device="cuda")
    H = torch.full((R * B,), -1, dtype=torch.int32, device="cuda")
    q_d, a_d = pir.from_u32(Q.reshape(-1)), pir.from_u32(np.ascontiguousarray(Q.T).reshape(-1))
    for _ in range(2):
        pir.qpadl_pir_answer_batch(db, q_d, out, path=1)
        pir.qpadl_pir_hint(db, a_d, H)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    exp = oracle.answer_batch(D, Q, threads=oracle.max_threads())
    assert np.array_equal(pir.as_u32(out).reshape(B, R), exp)
    assert np.array_equal(pir.as_u32(H).reshape(R, B), exp.T)
    db.close()
