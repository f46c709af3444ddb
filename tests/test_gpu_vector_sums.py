"""What centring the digits takes from every output comes back from the vectors' sums, one word per 2048 columns
of a vector: batches on pair tiles (three and four limbs) and on tiles of one SM, at the edges of those blocks."""
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


@pytest.mark.parametrize("pair", [1, 0])
@pytest.mark.parametrize("B", [3, 66, 150])   # 150: three 64-vector halves, four limbs where that is the faster form
@pytest.mark.parametrize("C", [1, 8, 250, 2040, 2047, 2048, 2049, 4096, 4097, 6151, 20480])
def test_blocks_of_columns(C, B, pair):
    R = 300
    D = inputs.db_digits(R, C, 256, seed=C)
    Q = inputs.uniform_u32(B * C, seed=C + B, tag=inputs.TAG_MISC).reshape(B, C)
    Q[1] = 0xFFFFFFFF
    db = pir.qpadl_pir_setup(pir.params(R, C, 64), torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, pair)
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_U8_MAX_BATCH, 0)
    out = torch.empty(B * R, dtype=torch.int32, device="cuda")
    for _ in range(2):   # the second call finds the scratch of the first
        pir.qpadl_pir_answer_batch(db, pir.from_u32(Q.reshape(-1)), out, path=1)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    assert np.array_equal(pir.as_u32(out).reshape(B, R), oracle.answer_batch(D, Q, threads=oracle.max_threads()))
    db.close()


@pytest.mark.parametrize("pair", [1, 0])
@pytest.mark.parametrize("B", [3, 66, 150])
@pytest.mark.parametrize("p", [2, 4, 16, 128])   # digits are centred by p / 2
@pytest.mark.parametrize("largest", [False, True])
def test_centre_follows_p(p, B, pair, largest):
    R, C = 270, 2100
    D = np.full((R, C), p - 1, dtype=np.uint8) if largest else inputs.db_digits(R, C, p, seed=p)
    Q = inputs.uniform_u32(B * C, seed=p + B, tag=inputs.TAG_MISC).reshape(B, C)
    db = pir.qpadl_pir_setup(pir.params(R, C, B, p=p), torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, pair)
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_U8_MAX_BATCH, 0)
    out = torch.empty(B * R, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_answer_batch(db, pir.from_u32(Q.reshape(-1)), out, path=1)
    H = torch.empty(R * B, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_hint(db, pir.from_u32(np.ascontiguousarray(Q.T).reshape(-1)), H)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    exp = oracle.answer_batch(D, Q, threads=oracle.max_threads())
    assert np.array_equal(pir.as_u32(out).reshape(B, R), exp)
    assert np.array_equal(pir.as_u32(H).reshape(R, B), exp.T)
    db.close()
