"""Z_p Responses on 256-wide pair tiles: batches at the edges of the groups of 32 columns that a tile's end works on, and
tiles cut into two to eight column ranges (a few row tiles, thousands of columns, at least four chunks of 512 each),
whose residues are added and reduced once more, for small, middle and the largest p."""
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


def _check(R, C, p, B, low=None):
    D = (inputs.db_digits(R, C, 256, seed=R + C).astype(np.int64) % p).astype(np.uint8) if low is None else np.full((R, C), min(p, 256) - 1, dtype=np.uint8)
    Q = (inputs.uniform_u32(B * C, seed=B + p, tag=inputs.TAG_MISC) % p).astype(np.uint32).reshape(B, C)
    if low is not None:
        Q[0] = low
    h = pir.qpadl_goldberg_setup(R, C, p, torch.from_numpy(D).cuda())
    out = torch.full((B * R,), -1, dtype=torch.int32, device="cuda")
    for _ in range(2):   # the second call adds to what the first one left, unless it is zeroed
        pir.qpadl_goldberg_answer_batch(h, pir.from_u32(Q.reshape(-1)), out)
    torch.cuda.synchronize()
    assert pir.qpadl_goldberg_status(h) == pir.QPADL_OK
    exp = oracle.goldberg_answer(D, Q, p, threads=oracle.max_threads())
    assert np.array_equal(pir.as_u32(out).reshape(B, R), exp)
    h.close()


@pytest.mark.parametrize("B", [129, 159, 160, 161, 192, 255, 256, 257, 288, 289, 385])
@pytest.mark.parametrize("R,C", [(1, 300), (257, 512), (300, 1100), (129, 1537)])
def test_groups_of_columns(R, C, B):
    _check(R, C, 257, B)


@pytest.mark.parametrize("R,C,B", [(300, 30001, 130), (257, 12289, 255), (200, 9000, 257), (100, 65536, 129), (600, 20011, 300)])
@pytest.mark.parametrize("p", [2, 3, 31, 251, 257])
def test_ranges_add_up(R, C, B, p):
    _check(R, C, p, B)


@pytest.mark.parametrize("p", [2, 257])
def test_ranges_of_the_largest_sums(p):   # centred entries of the largest magnitude against the largest digits
    _check(256, 16384, p, 130, low=p // 2)
    _check(256, 16384, p, 130, low=p // 2 + 1 if p > 2 else 1)
