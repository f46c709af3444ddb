"""Serving: the continuous-batching request loop over several resident
databases gives every request the same answer it gets alone, refuses
admission when memory or slots run out, and fails (rather than hangs)
requests whose completion never arrives (host-side fault injection).
"""
import time

import numpy as np
import pytest
import torch

import oracle
from paper_2510_03631_gb300 import inputs, pir

pytestmark = pytest.mark.gpu

SHAPES = [(512, 1024), (1000, 2048), (300, 4096 + 48)]   # ragged; the last one is not a multiple of 256


@pytest.fixture(scope="module")
def dbs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    out = []
    for k, (R, C) in enumerate(SHAPES):
        D = inputs.db_digits(R, C, 256, seed=50 + k)
        h = pir.qpadl_pir_setup(pir.params(R, C, 16, seed=50 + k), torch.from_numpy(D).cuda())
        out.append((D, h))
    yield out
    for _, h in out:
        h.close()


def _wait(srv, ticket, R, timeout=30.0):
    ans = np.zeros(R, dtype=np.uint32)
    t0 = time.time()
    while True:
        rc, times = pir.qpadl_server_poll(srv, ticket, ans)
        if rc != pir.QPADL_EAGAIN:
            return rc, ans, times
        if time.time() - t0 > timeout:
            raise AssertionError("request did not complete")
        time.sleep(0.0005)


def _server(dbs, **kw):
    srv = pir.qpadl_server_create(pir.server_config(**kw))
    ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
    pir.qpadl_server_start(srv)
    return srv, ids


def test_mixed_traffic_answers_equal_standalone(dbs):
    srv, ids = _server(dbs, max_batch=64, num_streams=3)
    rng = np.random.default_rng(7)
    which = [int(rng.choice(len(dbs), p=[0.6, 0.3, 0.1])) for _ in range(240)]
    qs = [inputs.uniform_u32(SHAPES[d][1], seed=1000 + i, tag=inputs.TAG_MISC) for i, d in enumerate(which)]
    reqs = []
    for i, (d, q) in enumerate(zip(which, qs)):
        reqs.append((d, q, pir.qpadl_server_submit(srv, ids[d], q)))
        if i % 37 == 0:
            time.sleep(0.002)   # let launches start while more requests arrive
    for d, q, t in reqs:
        D, h = dbs[d]
        rc, ans, times = _wait(srv, t, SHAPES[d][0])
        assert rc == pir.QPADL_OK
        # the same query answered alone, through the single-query entry point
        alone = torch.empty(SHAPES[d][0], dtype=torch.int32, device="cuda")
        pir.qpadl_pir_answer(h, pir.from_u32(q), alone)
        torch.cuda.synchronize()
        assert np.array_equal(ans, pir.as_u32(alone))
        assert times[0] <= times[1] <= times[2]
    st = pir.qpadl_server_stats(srv)
    assert st["completed"] == 240 and st["failed"] == 0 and st["inflight"] == 0
    # how many launches the burst takes depends on timing; batching itself is
    # pinned by the launch formed from requests queued before start
    assert 1 <= st["launches"] <= 240
    srv.close()


def test_answers_match_oracle(dbs):
    srv, ids = _server(dbs, max_batch=8, num_streams=2)
    tickets = []
    for d in range(len(dbs)):
        C = SHAPES[d][1]
        for i in range(5):
            q = inputs.uniform_u32(C, seed=77 + 10 * d + i, tag=inputs.TAG_MISC)
            tickets.append((d, q, pir.qpadl_server_submit(srv, ids[d], q)))
    for d, q, t in tickets:
        rc, ans, _ = _wait(srv, t, SHAPES[d][0])
        assert rc == pir.QPADL_OK
        assert np.array_equal(ans, oracle.answer(dbs[d][0], q))
    srv.close()


@pytest.mark.parametrize("counts", [(3, 20, 45), (2, 20, 45), (5, 17, 32), (1, 0, 3), (1, 1, 1), (0, 64, 0)])
def test_one_launch_answers_every_database(dbs, counts):
    # requests submitted before start form one launch over all databases, and that launch runs
    # ONE grouped GEMM kernel however uneven the counts (the streaming kernel only for a lone
    # database with one or two queries)
    srv = pir.qpadl_server_create(pir.server_config(max_batch=64, num_streams=1, group_size_ratio=1e9))
    ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
    tickets = []
    for d, cnt in enumerate(counts):
        C = SHAPES[d][1]
        for i in range(cnt):
            q = inputs.uniform_u32(C, seed=9000 + 100 * d + i, tag=inputs.TAG_MISC)
            tickets.append((d, q, pir.qpadl_server_submit(srv, ids[d], q)))
    pir.qpadl_server_start(srv)
    for d, q, t in tickets:
        rc, ans, _ = _wait(srv, t, SHAPES[d][0])
        assert rc == pir.QPADL_OK
        assert np.array_equal(ans, oracle.answer(dbs[d][0], q))
    st = pir.qpadl_server_stats(srv)
    assert st["launches"] == 1 and st["completed"] == sum(counts)
    assert st["grouped_launches"] == (1 if sum(c > 0 for c in counts) > 1 else 0)
    assert st["gemm_kernels"] == 1 and st["stream_kernels"] == 0
    srv.close()


def test_group_above_the_uint8_gemm_limit_takes_the_fp16_copy(dbs):
    # a handle whose uint8-digit GEMM takes at most 8 queries: 20 queued queries of it run the
    # fp16-copy GEMM, the other databases' queries the grouped uint8-digit GEMM, in one cycle
    D1, h1 = dbs[1]
    pir.qpadl_pir_set_option(h1, pir.QPADL_OPT_U8_MAX_BATCH, 8)
    try:
        srv = pir.qpadl_server_create(pir.server_config(max_batch=64, num_streams=1, group_size_ratio=1e9))
        ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
        tickets = []
        for d, cnt in enumerate((4, 20, 6)):
            for i in range(cnt):
                q = inputs.uniform_u32(SHAPES[d][1], seed=9500 + 100 * d + i, tag=inputs.TAG_MISC)
                tickets.append((d, q, pir.qpadl_server_submit(srv, ids[d], q)))
        pir.qpadl_server_start(srv)
        for d, q, t in tickets:
            rc, ans, _ = _wait(srv, t, SHAPES[d][0])
            assert rc == pir.QPADL_OK and np.array_equal(ans, oracle.answer(dbs[d][0], q))
        st = pir.qpadl_server_stats(srv)
        assert st["launches"] == 1 and st["gemm_kernels"] == 2 and st["stream_kernels"] == 0
        srv.close()
    finally:
        pir.qpadl_pir_set_option(h1, pir.QPADL_OPT_U8_MAX_BATCH, 64)


@pytest.mark.parametrize("d,count", [(0, 150), (1, 192), (2, 129), (0, 3)])
@pytest.mark.parametrize("pair", [1, 0])
def test_group_of_an_odd_number_of_64_query_halves(dbs, d, count, pair):
    # one launch of 129-192 queries on the fp16 copy, where four byte limbs and a sum per query can be the
    # faster form: the workspace of a group has room for them (the smallest group on the copy too)
    D, h = dbs[d]
    pir.qpadl_pir_set_option(h, pir.QPADL_OPT_PAIR_GEMM, pair)
    pir.qpadl_pir_set_option(h, pir.QPADL_OPT_U8_MAX_BATCH, 2)
    try:
        srv = pir.qpadl_server_create(pir.server_config(max_batch=256, num_streams=1, max_inflight=512,
                                                        host_budget_bytes=64 << 20))
        db_id = pir.qpadl_server_add_db(srv, h)
        Q = inputs.uniform_u32(count * SHAPES[d][1], seed=count + d, tag=inputs.TAG_MISC).reshape(count, -1)
        tickets = [pir.qpadl_server_submit(srv, db_id, q) for q in Q]
        pir.qpadl_server_start(srv)
        exp = oracle.answer_batch(D, Q, threads=oracle.max_threads())
        for b, t in enumerate(tickets):
            rc, ans, _ = _wait(srv, t, SHAPES[d][0])
            assert rc == pir.QPADL_OK and np.array_equal(ans, exp[b])
        st = pir.qpadl_server_stats(srv)
        assert st["launches"] == 1 and st["gemm_kernels"] == 1
        srv.close()
    finally:
        pir.qpadl_pir_set_option(h, pir.QPADL_OPT_U8_MAX_BATCH, 64)
        pir.qpadl_pir_set_option(h, pir.QPADL_OPT_PAIR_GEMM, 1)


@pytest.mark.parametrize("ratio,grouped", [(0.0, False), (1.5, False), (2.5, True)])
def test_group_size_ratio(dbs, ratio, grouped):
    # sizes R*C: 0.5M, 2M and 1.24M words; with ratio 2.5 databases 1 and 2 share a launch
    srv = pir.qpadl_server_create(pir.server_config(max_batch=64, num_streams=1, group_size_ratio=ratio))
    ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
    tickets = []
    for d in (1, 2):
        for i in range(4):
            q = inputs.uniform_u32(SHAPES[d][1], seed=7000 + 10 * d + i, tag=inputs.TAG_MISC)
            tickets.append((d, q, pir.qpadl_server_submit(srv, ids[d], q)))
    pir.qpadl_server_start(srv)
    for d, q, t in tickets:
        rc, ans, _ = _wait(srv, t, SHAPES[d][0])
        assert rc == pir.QPADL_OK and np.array_equal(ans, oracle.answer(dbs[d][0], q))
    st = pir.qpadl_server_stats(srv)
    assert st["launches"] == (1 if grouped else 2)
    assert st["grouped_launches"] == (1 if grouped else 0)
    srv.close()


def test_launch_shrinks_to_the_device_budget(dbs):
    # the device arena holds the workspace of only a few requests of database 1
    R, C = SHAPES[1]
    per = 4 * C + 4 * R + 8 * C   # query, answer and query limbs (C is a multiple of 8)
    srv = pir.qpadl_server_create(pir.server_config(max_batch=64, num_streams=2, device_budget_bytes=5 * per))
    ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
    qs = [inputs.uniform_u32(C, seed=300 + i, tag=inputs.TAG_MISC) for i in range(24)]
    tickets = [pir.qpadl_server_submit(srv, ids[1], q) for q in qs]
    pir.qpadl_server_start(srv)
    for q, t in zip(qs, tickets):
        rc, ans, _ = _wait(srv, t, R)
        assert rc == pir.QPADL_OK
        assert np.array_equal(ans, oracle.answer(dbs[1][0], q))
    assert pir.qpadl_server_stats(srv)["launches"] >= 24 // 5
    srv.close()


def test_admission_refuses_when_slots_run_out(dbs):
    # a long hold keeps requests queued so the in-flight limit is reached
    srv, ids = _server(dbs, max_inflight=4, max_batch=4, num_streams=1)
    C = SHAPES[0][1]
    tickets, refused = [], 0
    for i in range(12):
        try:
            tickets.append(pir.qpadl_server_submit(srv, ids[0], inputs.uniform_u32(C, seed=i, tag=7)))
        except pir.QpadlError as e:
            assert e.code == pir.QPADL_EBUSY
            refused += 1
    assert len(tickets) <= 4 and refused >= 8
    for t in tickets:
        assert _wait(srv, t, SHAPES[0][0])[0] == pir.QPADL_OK
    # slots free again after polling
    t = pir.qpadl_server_submit(srv, ids[0], inputs.uniform_u32(C, seed=99, tag=7))
    assert _wait(srv, t, SHAPES[0][0])[0] == pir.QPADL_OK
    assert pir.qpadl_server_stats(srv)["refused"] >= 8
    srv.close()


def test_admission_refuses_when_host_memory_runs_out(dbs):
    R, C = SHAPES[1]
    per_request = 4 * (R + C) + 512
    srv, ids = _server(dbs, host_budget_bytes=3 * per_request, max_inflight=100, num_streams=1)
    ok, busy = [], 0
    for i in range(10):
        try:
            ok.append(pir.qpadl_server_submit(srv, ids[1], inputs.uniform_u32(C, seed=i, tag=7)))
        except pir.QpadlError as e:
            assert e.code == pir.QPADL_EBUSY
            busy += 1
    assert 1 <= len(ok) <= 3 and busy >= 7
    for t in ok:
        assert _wait(srv, t, R)[0] == pir.QPADL_OK
    srv.close()


def test_bad_arguments(dbs):
    srv, ids = _server(dbs)
    with pytest.raises(pir.QpadlError) as e:
        pir.qpadl_server_submit(srv, 17, np.zeros(16, np.uint32))
    assert e.value.code == pir.QPADL_EINVAL
    rc, _ = pir.qpadl_server_poll(srv, 123456789)
    assert rc == pir.QPADL_EINVAL
    srv.close()
    with pytest.raises(pir.QpadlError):
        pir.qpadl_server_create(pir.server_config(max_batch=0))


def test_watchdog_fails_a_launch_whose_completion_never_arrives(dbs):
    # host-side fault injection: the first launch's completion is dropped
    srv, ids = _server(dbs, max_batch=4, num_streams=2, watchdog_ms=200.0, test_drop_completion_launch=1)
    R, C = SHAPES[0]
    t1 = pir.qpadl_server_submit(srv, ids[0], inputs.uniform_u32(C, seed=1, tag=7))
    rc, _, _ = _wait(srv, t1, R, timeout=10)
    assert rc == pir.QPADL_ETIMEOUT
    # later launches are unaffected
    q = inputs.uniform_u32(C, seed=2, tag=7)
    t2 = pir.qpadl_server_submit(srv, ids[0], q)
    rc, ans, _ = _wait(srv, t2, R)
    assert rc == pir.QPADL_OK and np.array_equal(ans, oracle.answer(dbs[0][0], q))
    assert pir.qpadl_server_stats(srv)["failed"] == 1
    srv.close()


def test_replay_open_loop(dbs):
    srv, ids = _server(dbs, max_batch=64, num_streams=4)
    n = 400
    arr = inputs.poisson_arrivals(20000.0, n, seed=3)
    which = inputs.skewed_choice(n, (0.6, 0.3, 0.1), seed=4)
    queries = [inputs.uniform_u32(SHAPES[d][1], seed=500 + i, tag=7) for i, d in enumerate(which)]
    answers = [np.zeros(SHAPES[d][0], dtype=np.uint32) for d in which]
    lat, st, tm = pir.qpadl_server_replay(srv, arr, [ids[d] for d in which], queries, answers, with_times=True)
    assert (st == pir.QPADL_OK).all()
    assert (lat > 0).all()
    # submit, launch and completion follow the scheduled arrival in order; latency is completion
    assert (tm[:, 0] >= -1e-6).all() and (tm[:, 1] >= tm[:, 0]).all() and (tm[:, 2] >= tm[:, 1]).all()
    assert np.allclose(tm[:, 2], lat)
    for i in range(0, n, 17):
        d = which[i]
        assert np.array_equal(answers[i], oracle.answer(dbs[d][0], queries[i]))
    srv.close()


def test_replay_rejects_unsorted_arrivals(dbs):
    srv, ids = _server(dbs)
    qs = [inputs.uniform_u32(SHAPES[0][1], seed=i, tag=7) for i in range(3)]
    with pytest.raises(pir.QpadlError) as e:
        pir.qpadl_server_replay(srv, np.array([0.0, 2e-3, 1e-3]), [ids[0]] * 3, qs)
    assert e.value.code == pir.QPADL_EINVAL
    srv.close()


@pytest.mark.parametrize("d", range(len(SHAPES)))
def test_two_queued_queries_share_one_scan(dbs, d):
    # two requests for one database, queued before start, form one launch whose
    # streaming kernel answers both in a single pass over the database
    srv = pir.qpadl_server_create(pir.server_config(max_batch=64, num_streams=1))
    ids = [pir.qpadl_server_add_db(srv, h) for _, h in dbs]
    R, C = SHAPES[d]
    tickets = []
    for i in range(2):
        q = inputs.uniform_u32(C, seed=4200 + 10 * d + i, tag=inputs.TAG_MISC)
        tickets.append((q, pir.qpadl_server_submit(srv, ids[d], q)))
    pir.qpadl_server_start(srv)
    for q, t in tickets:
        rc, ans, _ = _wait(srv, t, R)
        assert rc == pir.QPADL_OK
        assert np.array_equal(ans, oracle.answer(dbs[d][0], q))
    st = pir.qpadl_server_stats(srv)
    assert st["launches"] == 1 and st["completed"] == 2
    assert st["stream_kernels"] == 1 and st["gemm_kernels"] == 0
    srv.close()
