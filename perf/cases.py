"""Workloads of the PIR library as its users run them, for measuring speed.

Each case is a dict of plain sizes with a `kind`; `prepare` makes the inputs and
handles a program would hold, `run` makes one pass through the public entry
points, `work` counts the bytes and operations the pass cannot do without and
`exact` computes the same outputs in 64-bit arithmetic with torch and numpy.

kinds
  batch     Response of the lattice scheme: one query (qpadl_pir_answer) or a batch
  hint      the offline hint D A of a database
  online    Query -> Response -> Recover with the handle-free client calls
  client    Query and Recover of many secrets through a client context
  chor      Response over GF(2): records are rows of bits
  goldberg  Response over Z_p: records are columns of field elements
  compress  width, encoding and decoding of sorted entries stored as differences
  serve     a burst of requests to a server that holds two databases
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_03631_gb300 import pir

DEV = "cuda"


def listed():
    return [
        # the smallest Response: a 1 MiB table, where launches and latency are everything
        dict(name="answer_1mib", kind="batch", rows=1024, cols=1024, p=256, batch=1),
        # one query against the full 1 GiB database: the memory-bound scan
        dict(name="answer_1gib", kind="batch", rows=32768, cols=32768, p=256, batch=1),
        # a small server batch on the same database
        dict(name="batch32_1gib", kind="batch", rows=32768, cols=32768, p=256, batch=32),
        # many users at once: 256 concurrent queries
        dict(name="batch256_1gib", kind="batch", rows=32768, cols=32768, p=256, batch=256),
        # offline phase of that database at LWE dimension 1024
        dict(name="hint_1gib", kind="hint", rows=32768, cols=32768, p=256, n=1024),
        # a client's single retrieval on a 256 MiB database
        dict(name="online_256mib", kind="online", rows=16384, cols=16384, p=256, n=1024, batch=1),
        # a few retrievals on a table with no round dimension and 4-bit digits
        dict(name="online_ragged", kind="online", rows=5003, cols=7001, p=16, n=630, batch=24),
        # a proxy that makes and opens 1024 queries through one client context
        dict(name="client_1024", kind="client", rows=32768, cols=32768, p=256, n=1024, batch=1024),
        # XOR scheme, 2^18 records of 3 KB, 128 users
        dict(name="chor_128", kind="chor", rows=1 << 18, bits=24576, batch=128),
        # field scheme, 2^16 records of 3 KB, 1024 users
        dict(name="goldberg_1024", kind="goldberg", rows=3072, cols=1 << 16, p=257, batch=1024),
        # storing 2^26 sorted entries as differences, and a client opening 64 blocks
        dict(name="compress_256mib", kind="compress", entries=1 << 26, block=8192, max_gap=31, open=64),
        # 256 requests arriving together at a server with a 16 MiB and a 256 MiB database
        dict(name="serve_256", kind="serve", side0=4096, side1=16384, requests=256, share1=0.3),
    ]


def _size(rng, lo, hi, step=64):
    """A size spread over the logarithm of [lo, hi]; half of them whole multiples of `step`."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, v // step * step)) if rng.random() < 0.5 else v


def _matrix(rng, lo, cells):
    """Rows and columns from `lo` up, at most `cells` in all, spread over the logarithm of their product."""
    side = math.sqrt(math.exp(rng.uniform(math.log(lo * lo), math.log(cells))))
    skew = math.exp(rng.uniform(-1.0, 1.0))
    rows, cols = (max(lo, int(v)) for v in (side * skew, side / skew))
    rows, cols = (v if rng.random() < 0.5 else v // 64 * 64 for v in (rows, cols))
    return rows, min(cols, cells // rows)


def draw(rng):
    kind = rng.choice(["batch", "batch", "batch", "hint", "online", "online", "client", "chor", "chor", "goldberg",
                       "compress", "serve"])
    if kind == "batch":
        rows, cols = _matrix(rng, 512, 1 << 30)
        return dict(kind=kind, rows=rows, cols=cols, p=rng.choice([256, 256, 16, 2]), batch=_size(rng, 1, 512, 8) or 1)
    if kind == "hint":
        rows, cols = _matrix(rng, 512, 1 << 29)
        return dict(kind=kind, rows=rows, cols=cols, p=256, n=rng.choice([512, 630, 1024, 1024, 2048]))
    if kind == "online":
        rows, cols = _matrix(rng, 512, 1 << 29)
        return dict(kind=kind, rows=rows, cols=cols, p=rng.choice([256, 256, 16]), n=rng.choice([512, 630, 1024, 2048]),
                    batch=rng.choice([1, 1, 2, _size(rng, 3, 128, 8)]))
    if kind == "client":
        rows, cols = _size(rng, 512, 32768), _size(rng, 512, 32768)
        return dict(kind=kind, rows=rows, cols=cols, p=256, n=rng.choice([512, 630, 1024]),
                    batch=_size(rng, 8, 1024, 32))
    if kind == "chor":
        rows = _size(rng, 1 << 10, 1 << 18)
        bits = 128 * _size(rng, 4, max(5, min(192, (1 << 32) // (128 * rows))), 8)
        return dict(kind=kind, rows=rows, bits=bits, batch=_size(rng, 1, 1024 if rows <= 1 << 16 else 256, 8))
    if kind == "goldberg":
        rows = _size(rng, 256, 8192)
        return dict(kind=kind, rows=rows, cols=_size(rng, 1024, 65536), p=rng.choice([257, 257, 251, 31]),
                    batch=_size(rng, 1, 1024, 8))
    if kind == "compress":
        return dict(kind=kind, entries=_size(rng, 1 << 16, 1 << 26, 4096), block=rng.choice([512, 1000, 4096, 8192]),
                    max_gap=rng.choice([31, 31, 2000]), open=rng.choice([1, 8, 64]))
    return dict(kind=kind, side0=_size(rng, 1024, 4096), side1=_size(rng, 4096, 16384), requests=_size(rng, 16, 512, 8),
                share1=round(rng.uniform(0.1, 0.5), 2))


# ---------------------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _digits(g, rows, cols, p):
    return torch.randint(0, p, (rows, cols), dtype=torch.uint8, device=DEV, generator=g)


def _words(g, *shape):
    """Uniform 32-bit words (the bits of int32)."""
    return torch.randint(-(1 << 31), 1 << 31, shape, dtype=torch.int32, device=DEV, generator=g)


def _noise(g, *shape):
    """Rounded Gaussian noise of standard deviation 6.4."""
    return (torch.randn(shape, device=DEV, generator=g) * 6.4).round().to(torch.int32)


def _targets(g, batch, cols):
    return torch.randint(0, cols, (batch,), dtype=torch.int32, device=DEV, generator=g)


def _inputs(case, seed):
    """Every tensor of the case, from the seed alone."""
    g, k = _gen(seed), case["kind"]
    if k == "batch":
        return dict(D=_digits(g, case["rows"], case["cols"], case["p"]), Q=_words(g, case["batch"], case["cols"]))
    if k == "hint":
        return dict(D=_digits(g, case["rows"], case["cols"], case["p"]), A=_words(g, case["cols"], case["n"]))
    if k in ("online", "client"):
        R, C, n, B = case["rows"], case["cols"], case["n"], case["batch"]
        x = dict(A=_words(g, C, n), H=_words(g, R, n), S=_words(g, B, n), E=_noise(g, B, C), cols=_targets(g, B, C))
        if k == "online":
            x["D"] = _digits(g, R, C, case["p"])
        else:
            x["ans"] = _words(g, B, R)
        return x
    if k == "chor":
        Q = _words(g, case["batch"], (case["rows"] + 31) // 32)
        return dict(D=_words(g, case["rows"], case["bits"] // 32), Q=Q)
    if k == "goldberg":
        p = case["p"]
        return dict(D=_digits(g, case["rows"], case["cols"], min(p, 256)),
                    Q=torch.randint(0, p, (case["batch"], case["cols"]), dtype=torch.int32, device=DEV, generator=g))
    if k == "compress":
        gaps = torch.randint(0, case["max_gap"] + 1, (case["entries"],), dtype=torch.int32, device=DEV, generator=g)
        return dict(x=torch.cumsum(gaps, 0, dtype=torch.int32))
    D = [_digits(g, s, s, 256) for s in (case["side0"], case["side1"])]
    ids = (torch.randperm(case["requests"], device=DEV, generator=g) < int(case["requests"] * case["share1"]))
    ids = ids.cpu().numpy().astype(np.int32)
    Q = [_words(g, int((ids == i).sum()), s).cpu().numpy().view(np.uint32)
         for i, s in enumerate((case["side0"], case["side1"]))]
    return dict(D=D, ids=ids, Q=Q)


def _pad_blocks(x, E):
    """The entries as whole blocks, positions past the end repeating the last entry (int64, blocks x E)."""
    pad = -x.numel() % E
    v = torch.cat([x, x[-1:].expand(pad)]) if pad else x
    return v.reshape(-1, E).to(torch.int64)


def _width(d):
    m = int(d.max()) if d.numel() else 0
    return next(w for w in (1, 2, 3, 4) if w == 4 or m < 1 << (8 * w))


def _block_digits(v, w):
    """Stored digits of blocks of entries, one block per row: 4 bytes of the first, then w bytes a difference."""
    byte = lambda t, k: ((t >> (8 * k)) & 255).to(torch.uint8)
    first = torch.stack([byte(v[:, 0], k) for k in range(4)], 1)
    d = (v[:, 1:] - v[:, :-1]) & 0xFFFFFFFF
    return torch.cat([first, torch.stack([byte(d, k) for k in range(w)], 2).reshape(v.shape[0], -1)], 1)


def prepare(case, seed):
    x, k = _inputs(case, seed), case["kind"]
    empty = lambda *shape, t=torch.int32: torch.empty(shape, dtype=t, device=DEV)
    st = dict(x, kind=k, case=case)
    if k in ("batch", "hint", "online"):
        prm = pir.params(case["rows"], case["cols"], case.get("n", 1024), p=case["p"], seed=seed)
        st["prm"], st["db"] = prm, pir.qpadl_pir_setup(prm, x["D"])
        if k != "hint":
            pir.qpadl_pir_reserve(st["db"], case["batch"])
            st["ans"] = empty(case["batch"], case["rows"])
        else:
            st["H"] = empty(case["rows"], case["n"])
        if k == "online":
            st.update(q=empty(case["batch"], case["cols"]), out=empty(case["batch"], case["rows"], t=torch.uint8),
                      col=int(x["cols"][0]))
    elif k == "client":
        prm = pir.params(case["rows"], case["cols"], case["n"], p=case["p"], seed=seed)
        st.update(ctx=pir.qpadl_client_create(prm, x["A"], x["H"], max_batch=case["batch"]),
                  q=empty(case["batch"], case["cols"]), out=empty(case["batch"], case["rows"], t=torch.uint8))
    elif k == "chor":
        st.update(db=pir.qpadl_chor_setup(case["rows"], case["bits"], x["D"]),
                  out=empty(case["batch"], case["bits"] // 32))
    elif k == "goldberg":
        st.update(db=pir.qpadl_goldberg_setup(case["rows"], case["cols"], case["p"], x["D"]),
                  out=empty(case["batch"], case["rows"]))
    elif k == "compress":
        E = case["block"]
        opened = min(case["open"], case["entries"] // E)
        w = 1 if case["max_gap"] < 256 else 2
        st.update(w_open=w, digits=_block_digits(_pad_blocks(x["x"][: opened * E], E), w).contiguous(),
                  opened=opened, entries=empty(opened, E))
    else:
        sides = (case["side0"], case["side1"])
        need = 8 * sum(q.shape[0] * s for q, s in zip(x["Q"], sides))
        srv = pir.qpadl_server_create(pir.server_config(host_budget_bytes=max(32 << 20, 2 * need),
                                                        device_budget_bytes=512 << 20))
        for s, D in zip(sides, x["D"]):
            pir.qpadl_server_add_db(srv, pir.qpadl_pir_setup(pir.params(s, s, 1024, seed=seed), D))
        pir.qpadl_server_start(srv)
        st["srv"], at = srv, [0, 0]
        st["answers"] = [np.zeros((q.shape[0], s), np.uint32) for q, s in zip(x["Q"], sides)]
        st["queries"], st["slots"] = [], []
        for i in x["ids"]:
            st["queries"].append(x["Q"][i][at[i]])
            st["slots"].append(st["answers"][i][at[i]])
            at[i] += 1
        st["arrivals"] = np.zeros(len(x["ids"]))
    return st


def run(st):
    k = st["kind"]
    if k == "batch":
        if st["Q"].shape[0] == 1:
            return pir.qpadl_pir_answer(st["db"], st["Q"], st["ans"])
        return pir.qpadl_pir_answer_batch(st["db"], st["Q"], st["ans"])
    if k == "hint":
        return pir.qpadl_pir_hint(st["db"], st["A"], st["H"])
    if k == "online":
        if st["S"].shape[0] == 1:
            pir.qpadl_pir_query(st["prm"], st["A"], st["S"], st["E"], st["col"], st["q"])
            pir.qpadl_pir_answer(st["db"], st["q"], st["ans"])
            pir.qpadl_pir_recover(st["prm"], st["ans"], st["H"], st["S"], st["out"])
        else:
            pir.qpadl_pir_query_batch(st["prm"], st["A"], st["S"], st["E"], st["cols"], st["q"])
            pir.qpadl_pir_answer_batch(st["db"], st["q"], st["ans"])
            pir.qpadl_pir_recover_batch(st["prm"], st["ans"], st["H"], st["S"], st["out"])
        return st["q"], st["ans"], st["out"]
    if k == "client":
        pir.qpadl_client_query_batch(st["ctx"], st["S"], st["E"], st["cols"], st["q"])
        pir.qpadl_client_recover_batch(st["ctx"], st["ans"], st["S"], st["out"])
        return st["q"], st["out"]
    if k == "chor":
        return pir.qpadl_chor_answer_batch(st["db"], st["Q"], st["out"])
    if k == "goldberg":
        return pir.qpadl_goldberg_answer_batch(st["db"], st["Q"], st["out"])
    if k == "compress":
        x, E = st["x"], st["case"]["block"]
        w = pir.qpadl_pir_delta_width(x, E)
        db = torch.empty(pir.delta_rows(E, w), -(-x.numel() // E), dtype=torch.uint8, device=x.device)
        pir.qpadl_pir_delta_encode(x, E, w, db)
        pir.qpadl_pir_delta_decode(st["digits"], st["opened"], E, st["w_open"], st["entries"])
        return w, db, st["entries"]
    _, status = pir.qpadl_server_replay(st["srv"], st["arrivals"], st["ids"], st["queries"], st["slots"])
    return status, st["answers"]


def work(case):
    k = case["kind"]
    if k in ("batch", "goldberg"):
        R, C, B = case["rows"], case["cols"], case["batch"]
        return dict(bytes=R * C + 4 * B * (C + R), flops=2 * R * C * B)
    if k == "hint":
        R, C, n = case["rows"], case["cols"], case["n"]
        return dict(bytes=R * C + 4 * n * (C + R), flops=2 * R * C * n)
    if k in ("online", "client"):
        R, C, n, B = case["rows"], case["cols"], case["n"], case["batch"]
        b, f = 4 * n * (C + R + B) + 8 * B * C + 5 * B * R, 2 * B * n * (C + R)
        return dict(bytes=b + R * C, flops=f + 2 * R * C * B) if k == "online" else dict(bytes=b, flops=f)
    if k == "chor":
        W, B = case["bits"] // 32, case["batch"]
        return dict(bytes=4 * (case["rows"] * W + B * ((case["rows"] + 31) // 32 + W)), flops=2 * case["rows"] * W * B)
    if k == "compress":
        n, w = case["entries"], 1 if case["max_gap"] < 256 else 2
        return dict(bytes=4 * n + w * n + case["open"] * case["block"] * (w + 4), flops=2 * n)
    n1 = int(case["requests"] * case["share1"])
    per = ((case["requests"] - n1, case["side0"]), (n1, case["side1"]))
    return dict(bytes=sum(s * s + 8 * n * s for n, s in per), flops=sum(2 * n * s * s for n, s in per))


# ---------------------------------------------------------------------------- 64-bit references
def _u32(t):
    return t.to(torch.int64) & 0xFFFFFFFF


def _mul_digits(D, X):
    """X D^T mod 2^32 for digits D (R x C) and 32-bit words X (B x C): exact products of 16-bit halves in float64."""
    x, out = _u32(X), []
    lo, hi = (x & 0xFFFF).double(), (x >> 16).double()
    for r in range(0, D.shape[0], 4096):
        d = D[r:r + 4096].double().t()
        out.append(((lo @ d).to(torch.int64) + (((hi @ d).to(torch.int64) & 0xFFFF) << 16)) & 0xFFFFFFFF)
    return torch.cat(out, 1)


def _mul_words(X, S):
    """S X^T mod 2^32 for 32-bit words X (R x n) and S (B x n)."""
    s, x = _u32(S), _u32(X)
    sl, sh = (s & 0xFFFF).double(), (s >> 16).double()
    xl, xh = (x & 0xFFFF).double().t(), (x >> 16).double().t()
    mid = (sl @ xh).to(torch.int64) + (sh @ xl).to(torch.int64)
    return ((sl @ xl).to(torch.int64) + ((mid & 0xFFFF) << 16)) & 0xFFFFFFFF


def _as_i32(t):
    return torch.where(t >= 1 << 31, t - (1 << 32), t).to(torch.int32)


def _recover(ans, H, S, p):
    shift = 32 - (p.bit_length() - 1)
    x = (ans - _mul_words(H, S) + (1 << (shift - 1))) & 0xFFFFFFFF
    return (x >> shift).to(torch.uint8)


def _bits(words):
    """Bits of the words of each row, lowest first (float64)."""
    s = torch.arange(32, device=words.device, dtype=torch.int32)
    return ((words.unsqueeze(-1) >> s) & 1).reshape(words.shape[0], -1).double()


def exact(case, seed):
    x, k = _inputs(case, seed), case["kind"]
    if k == "batch":
        return _as_i32(_mul_digits(x["D"], x["Q"]))
    if k == "hint":
        return _as_i32(_mul_digits(x["D"], x["A"].t())).t().contiguous()
    if k in ("online", "client"):
        q = _mul_words(x["A"], x["S"]) + x["E"]
        b = torch.arange(case["batch"], device=DEV)
        q[b, x["cols"].long()] += (1 << 32) // case["p"]
        q = q & 0xFFFFFFFF
        if k == "client":
            return _as_i32(q), _recover(_u32(x["ans"]), x["H"], x["S"], case["p"])
        ans = _mul_digits(x["D"], q)
        return _as_i32(q), _as_i32(ans), _recover(ans, x["H"], x["S"], case["p"])
    if k == "chor":
        R, W, q, out = case["rows"], case["bits"] // 32, _bits(x["Q"])[:, : case["rows"]], []
        pow2 = 1 << torch.arange(32, device=DEV, dtype=torch.int64)
        for c in range(0, W, 64):
            acc = 0
            for r in range(0, R, 1 << 16):
                acc = acc + q[:, r:r + (1 << 16)] @ _bits(x["D"][r:r + (1 << 16), c:c + 64])
            par = (acc.to(torch.int64) & 1).reshape(case["batch"], -1, 32)
            out.append(_as_i32((par * pow2).sum(2)))
        return torch.cat(out, 1)
    if k == "goldberg":
        return ((x["Q"].double() @ x["D"].double().t()).to(torch.int64) % case["p"]).to(torch.int32)
    if k == "compress":
        E = case["block"]
        v = _pad_blocks(x["x"], E)
        w = _width((v[:, 1:] - v[:, :-1]) & 0xFFFFFFFF)
        opened = min(case["open"], case["entries"] // E)
        return w, _block_digits(v, w).t().contiguous(), x["x"][: opened * E].reshape(opened, E)
    answers = []
    for D, Q in zip(x["D"], x["Q"]):
        q = torch.from_numpy(Q.view(np.int32)).to(DEV)
        answers.append(_mul_digits(D, q).cpu().numpy().astype(np.uint32) if Q.shape[0] else np.zeros((0, D.shape[0]), np.uint32))
    return np.zeros(case["requests"], np.int32), answers
