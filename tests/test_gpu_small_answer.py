"""One and two queries on small databases, where the streaming kernel packs them in the same launch
by default: equal to the oracle around the limits of that rule, for aligned and unaligned queries, and right
after a kernel that rewrites the database."""
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


# below, at and above 4096 columns, 4 Mi and 16 Mi digits; columns a multiple of 256, of 16, of neither
@pytest.mark.parametrize("R,C", [(1, 16), (9, 272), (1024, 1024), (1000, 4096), (300, 4112), (1024, 4096), (1025, 4096),
                                 (4096, 4096), (4097, 4096), (40000, 256), (77, 1001)])
@pytest.mark.parametrize("B,offset", [(1, 0), (1, 1), (2, 0), (2, 1)])
def test_answer(R, C, B, offset):
    D = inputs.db_digits(R, C, 256, seed=R + C)
    Q = inputs.uniform_u32(B * C, seed=R + B, tag=inputs.TAG_MISC).reshape(B, C)
    db = pir.qpadl_pir_setup(pir.params(R, C, 64), torch.from_numpy(D).cuda())
    buf = torch.zeros(B * C + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = pir.from_u32(Q.reshape(-1))
    out = torch.empty(B * R, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_answer_batch(db, buf[offset:], out)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    assert pir.qpadl_pir_get_option(db, pir.QPADL_OPT_STREAM_RAW) == 0
    assert np.array_equal(pir.as_u32(out).reshape(B, R), oracle.answer_batch(D, Q, threads=oracle.max_threads()))
    db.close()


def test_answer_follows_the_kernel_that_writes_the_database():
    R = C = 2048
    D_dev = torch.zeros(R * C, dtype=torch.uint8, device="cuda")
    db = pir.qpadl_pir_setup(pir.params(R, C, 64), D_dev)
    q = inputs.uniform_u32(C, seed=3, tag=inputs.TAG_MISC)
    q_d, out = pir.from_u32(q), torch.empty(R, dtype=torch.int32, device="cuda")
    for seed in range(4):
        D = inputs.db_digits(R, C, 256, seed=seed)
        src = torch.from_numpy(D).cuda().reshape(-1)
        torch.cuda.synchronize()
        torch.add(src, 0, out=D_dev)
        pir.qpadl_pir_answer(db, q_d, out)
        torch.cuda.synchronize()
        assert np.array_equal(pir.as_u32(out), oracle.answer(D, q))
    db.close()
