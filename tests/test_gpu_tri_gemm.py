"""Three-limb pair GEMM (batched Response and hint beyond the uint8-digit GEMM) equals the oracle bit
for bit: edges of its vector groups, tiles and 128-column exact chunks, tiles cut into column ranges,
and the values at the bound of the exact sums."""
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


def _setup(D, n=64, p=256):
    R, C = D.shape
    db = pir.qpadl_pir_setup(pir.params(R, C, n, p=p), torch.from_numpy(D).cuda())
    pir.qpadl_pir_set_option(db, pir.QPADL_OPT_U8_MAX_BATCH, 0)   # every batch takes the GEMM over the fp16 copy
    return db


def _answers(db, Q, R):
    out = torch.full((Q.shape[0] * R,), 0x55, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_answer_batch(db, pir.from_u32(np.ascontiguousarray(Q).reshape(-1)), out, path=1)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    return pir.as_u32(out).reshape(Q.shape[0], R)


# (R, C, B): one to many vector groups of 32, halves of 64, tiles of 128; columns around 64 and 128;
# long rows of few tiles (cut into ranges); more tiles than clusters
SHAPES = [(1, 1, 1), (255, 63, 31), (256, 64, 32), (257, 65, 33), (300, 127, 64), (513, 128, 65), (129, 129, 127),
          (700, 255, 128), (260, 1000, 129), (300, 1500, 192), (200, 1029, 193), (300, 5000, 40), (520, 8200, 200),
          (100, 20000, 130), (22000, 300, 70), (9000, 2048, 330),
          (20100, 200, 320), (700, 66000, 150), (300, 131200, 66), (257, 900, 449)]


@pytest.mark.parametrize("R,C,B", SHAPES)
def test_batched_response(R, C, B):
    D = inputs.db_digits(R, C, 256, seed=R + C)
    Q = inputs.uniform_u32(B * C, seed=B + C, tag=inputs.TAG_MISC).reshape(B, C)
    db = _setup(D)
    assert np.array_equal(_answers(db, Q, R), oracle.answer_batch(D, Q, threads=oracle.max_threads()))
    db.close()


@pytest.mark.parametrize("R,C,n", [(200, 300, 33), (300, 1000, 100), (520, 2100, 512), (257, 131, 70), (2000, 700, 130),
                                   (600, 700, 512), (300, 5000, 68), (9000, 200, 96), (700, 4000, 320)])
def test_hint(R, C, n):
    D = inputs.db_digits(R, C, 256, seed=R + n)
    A = inputs.public_matrix(C, n, seed=C)
    db = _setup(D, n)
    H = torch.empty(R * n, dtype=torch.int32, device="cuda")
    pir.qpadl_pir_hint(db, pir.from_u32(A.reshape(-1)), H)
    torch.cuda.synchronize()
    assert pir.qpadl_pir_status(db) == pir.QPADL_OK
    assert np.array_equal(pir.as_u32(H).reshape(R, n), oracle.hint(D, A, threads=oracle.max_threads()))
    db.close()


LIMB_MIN = (-1024 - (1024 << 11) - (512 << 22)) & 0xFFFFFFFF   # every balanced limb at its least
LIMB_MAX = (1023 + (1023 << 11) + (511 << 22)) & 0xFFFFFFFF


@pytest.mark.parametrize("digit", [0, 1, 128, 255])
@pytest.mark.parametrize("word", [LIMB_MIN, LIMB_MAX, 0, 0xFFFFFFFF, 1 << 10, 1 << 21, 1 << 31])
def test_bound_of_the_exact_sums(digit, word):
    # a constant row against a constant vector: a chunk's sum is 128 (d - 128) limb, up to 2^24 in
    # magnitude; the other rows and vectors alternate signs
    R, C, B = 260, 1024 + 17, 66
    D = np.full((R, C), digit, dtype=np.uint8)
    D[1::2, ::3] = 255 - digit
    Q = np.full((B, C), word, dtype=np.uint32)
    Q[1::2, ::5] = LIMB_MAX
    Q[2::4, 1::2] = LIMB_MIN
    db = _setup(D)
    assert np.array_equal(_answers(db, Q, R), oracle.answer_batch(D, Q, threads=oracle.max_threads()))
    db.close()


def test_option_changed_after_the_copy_was_made():
    R, C, B = 300, 700, 70
    D = inputs.db_digits(R, C, 256, seed=5)
    Q = inputs.uniform_u32(B * C, seed=6, tag=inputs.TAG_MISC).reshape(B, C)
    db, exp = _setup(D), oracle.answer_batch(D, Q, threads=oracle.max_threads())
    for pair in (1, 0, 1):
        pir.qpadl_pir_set_option(db, pir.QPADL_OPT_PAIR_GEMM, pair)
        assert np.array_equal(_answers(db, Q, R), exp)
    db.close()
