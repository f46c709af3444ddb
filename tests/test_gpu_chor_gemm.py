"""Chor Response on the tensor cores at the edges of its tiles: rows around a unit of 256 and around
the 2^18 rows of one launch, words around a column tile of 16, batches around 32, 64 and 128 query
tiles; all-ones databases and queries (the largest counts); the default choice of kernel by record
length.  Every answer equals the oracle's bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_03631_gb300 import inputs, pir

pytestmark = pytest.mark.gpu


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint32).view(np.int32).reshape(-1)).cuda()


def _check(rows, bits, B, DB, Q, min_batch):
    h = pir.qpadl_chor_setup(rows, bits, _dev(DB))
    if min_batch:
        pir.qpadl_chor_set_option(h, pir.QPADL_CHOR_OPT_M4RM_MIN_BATCH, min_batch)
    out = torch.empty(B * h.words, dtype=torch.int32, device="cuda")
    pir.qpadl_chor_answer_batch(h, _dev(Q), out)
    assert pir.qpadl_chor_status(h) == pir.QPADL_OK
    exp = oracle.chor_answer(DB, rows, Q, threads=oracle.max_threads())
    assert np.array_equal(pir.as_u32(out).reshape(B, h.words), exp)
    h.close()


@pytest.mark.parametrize("rows", [1, 31, 255, 256, 257, 1025])
@pytest.mark.parametrize("bits", [128, 512, 640, 4096 + 128])
@pytest.mark.parametrize("B", [1, 32, 33, 64, 65, 128, 129])
def test_tile_edges(rows, bits, B):
    _check(rows, bits, B, inputs.chor_db(rows, bits, seed=rows + bits), inputs.chor_queries(B, rows, seed=rows * 3 + B), 1)


@pytest.mark.parametrize("rows,B", [((1 << 18) - 1, 2), (1 << 18, 40), ((1 << 18) + 300, 70)])
def test_rows_of_one_launch(rows, B):
    _check(rows, 128, B, inputs.chor_db(rows, 128, seed=1), inputs.chor_queries(B, rows, seed=2), 1)


@pytest.mark.parametrize("rows,B", [(257, 33), (1 << 18, 3), (262143, 65)])
def test_largest_counts(rows, B):
    DB = np.full((rows, 4), 0xFFFFFFFF, np.uint32)
    Q = np.full((B, (rows + 31) // 32), 0xFFFFFFFF, np.uint32)
    _check(rows, 128, B, DB, Q, 1)


@pytest.mark.parametrize("bits", [511 * 32 // 128 * 128, 512 * 32, 1024 * 32])
@pytest.mark.parametrize("B", [1, 2, 3, 8, 9, 137])
def test_default_choice(bits, B):
    rows = 300
    _check(rows, bits, B, inputs.chor_db(rows, bits, seed=bits), inputs.chor_queries(B, rows, seed=B), None)


@pytest.mark.parametrize("min_batch,B", [(129, 128), (200, 199), (200, 256), (200, 330), (256, 256), (3, 258)])
def test_threshold_decides_for_chunks_of_256(min_batch, B):
    rows, bits = 700, 2048
    _check(rows, bits, B, inputs.chor_db(rows, bits, seed=B), inputs.chor_queries(B, rows, seed=min_batch), min_batch)


def test_option_reads_as_the_threshold_in_force():
    for bits, own in ((128, 1), (511 * 32 // 128 * 128, 1), (512 * 32, 3), (1023 * 32 // 128 * 128, 3), (1024 * 32, 9)):
        h = pir.qpadl_chor_setup(64, bits, _dev(np.zeros((64, bits // 32))))
        opt = lambda: pir.qpadl_chor_get_option(h, pir.QPADL_CHOR_OPT_M4RM_MIN_BATCH)
        assert opt() == own
        pir.qpadl_chor_set_option(h, pir.QPADL_CHOR_OPT_SCAN_FORM, 1)
        assert opt() == 48
        pir.qpadl_chor_set_option(h, pir.QPADL_CHOR_OPT_SCAN_FORM, -1)
        pir.qpadl_chor_set_option(h, pir.QPADL_CHOR_OPT_M4RM_MIN_BATCH, 200)
        assert opt() == 200
        h.close()


# several tiles of 128 queries in one launch, the last one whole, wide or narrow; more tiles than the scratch holds
# (eight up to 512 rows, two from 1400 and one from 2^17 on); a narrow rest in a launch of its own (more than 4096 units x column tiles)
@pytest.mark.parametrize("rows,bits,B", [(1, 128, 257), (300, 640, 129), (300, 640, 192), (300, 4096, 300), (2805, 1152, 190),
                                         (700, 1280, 726), (257, 512, 1025), (33000, 128, 300), (5000, 256, 700), (20000, 40960, 130), (1024, 16384, 129),
                                         ((1 << 18) + 700, 128, 140)])
@pytest.mark.parametrize("min_batch", [None, 1])
def test_tiles_of_one_launch(rows, bits, B, min_batch):
    _check(rows, bits, B, inputs.chor_db(rows, bits, seed=rows + B), inputs.chor_queries(B, rows, seed=B), min_batch)


# few rows of long records: XOR tables of four rows (chunks of 256, a short last one), and the scan up to 16 queries
@pytest.mark.parametrize("rows", [1, 63, 64, 65, 255, 256, 257])
@pytest.mark.parametrize("bits,B", [(2048 * 32, 64), (2048 * 32 + 128, 129), (4096 * 32, 33), (4096 * 32, 290), (8192 * 32, 16),
                                    (8192 * 32 + 1920, 17)])
def test_few_rows_of_long_records(rows, bits, B):
    _check(rows, bits, B, inputs.chor_db(rows, bits, seed=rows + B), inputs.chor_queries(B, rows, seed=bits), None)
