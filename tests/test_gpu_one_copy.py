"""A lattice handle keeps one fp16 copy of its digits, minus 128, that tiles over pairs of SMs and tiles of one SM
both read: after a reserve or the setup flag, changing the tile option builds nothing, also under capture, and the
answers and hints equal the oracle's either way."""
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


def _capture(fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        fn()
    return g


@pytest.mark.parametrize("flag", [0, 1])
@pytest.mark.parametrize("first", [1, 0])
def test_option_changed_after_reserve_under_capture(flag, first):
    R, C, B, n = 700, 1500, 150, 100
    D = inputs.db_digits(R, C, 256, seed=11)
    Q, A = inputs.uniform_u32(B * C, seed=12, tag=inputs.TAG_MISC).reshape(B, C), inputs.public_matrix(C, n, seed=13)
    prm = pir.params(R, C, n)
    prm.flags = flag
    db = pir.qpadl_pir_setup(prm, torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, first)
    pir.qpadl_pir_reserve(db, B)
    held = pir.qpadl_pir_device_bytes(db)
    q_d, a_d = pir.from_u32(Q.reshape(-1)), pir.from_u32(A.reshape(-1))
    out = torch.empty(B * R, dtype=torch.int32, device="cuda")
    H = torch.empty(R * n, dtype=torch.int32, device="cuda")
    exp, exp_h = oracle.answer_batch(D, Q, threads=oracle.max_threads()), oracle.hint(D, A, threads=oracle.max_threads())
    for pair in (1 - first, first):
        pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, pair)
        g = _capture(lambda: pir.qpadl_pir_answer_batch(db, q_d, out))
        h = _capture(lambda: pir.qpadl_pir_hint(db, a_d, H))
        for graph in (g, h):
            graph.replay()
        torch.cuda.synchronize()
        assert pir.qpadl_pir_status(db) == pir.QPADL_OK
        assert np.array_equal(pir.as_u32(out).reshape(B, R), exp)
        assert np.array_equal(pir.as_u32(H).reshape(R, n), exp_h)
    assert pir.qpadl_pir_device_bytes(db) == held
    db.close()


# single-SM tiles of 8, 16, 32 and 64 vectors; whole tiles, tiles split by chunks of 512 columns, ragged columns;
# vectors of more than 65536 columns, whose sums several blocks add up
@pytest.mark.parametrize("R,C,B", [(1, 1, 1), (129, 511, 3), (300, 1537, 16), (1000, 2048, 33), (20100, 520, 65),
                                   (400, 66001, 70)])
@pytest.mark.parametrize("digit", [None, 0, 255])
def test_single_sm_tiles(R, C, B, digit):
    D = inputs.db_digits(R, C, 256, seed=R) if digit is None else np.full((R, C), digit, dtype=np.uint8)
    Q = inputs.uniform_u32(B * C, seed=C + B, tag=inputs.TAG_MISC).reshape(B, C)
    Q[0] = 0x7F7F7F80   # byte limbs -128, -128, -128 and -128 (a carry each)
    db = pir.qpadl_pir_setup(pir.params(R, C, B), torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, 0)
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
