"""Check- and variable-node updates at every row and column width: random
irregular matrices against the FP32 oracle.  Both sides round every operation
alike, so posteriors, flip counts and results must be equal, not close."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from oracle import Code, Params as OParams  # noqa: E402
from paper_2507_00254_gb300 import bpsf as B  # noqa: E402
from paper_2507_00254_gb300 import codes, harness  # noqa: E402

pytestmark = pytest.mark.gpu

THREADS = max(1, min(16, os.cpu_count() or 1))


def irregular(rng, m, n, dc, dv):
    """Row degrees 2..dc (at least one row of each end), column degrees at most dv (0 among them)."""
    h = np.zeros((m, n), dtype=np.uint8)
    for j in range(m):
        want = dc if j == 0 else (2 if j == 1 else int(rng.integers(2, dc + 1)))
        free = np.nonzero(h.sum(axis=0) < dv)[0]
        h[j, rng.choice(free, size=min(want, free.size), replace=False)] = 1
    return h


def regular(rng, m, dc=6, dv=3):
    """Exactly dc ones per row and dv per column: shifted identities, columns shuffled."""
    n = m * dc // dv
    h = np.zeros((m, n), dtype=np.uint8)
    for i in range(n):
        for k in range(dv):
            h[(i + k * (k + 3) // 2 + k * (i // m)) % m, i] = 1
    return h[:, rng.permutation(n)]


CASES = [(dc, dv, s, lay, alpha) for dc, dv in ((2, 3), (3, 4), (5, 4), (6, 2), (7, 4), (8, 3), (9, 5), (10, 8), (16, 8),
                                                 (17, 9), (32, 16))
         for s, lay, alpha in ((1, False, 0.625), (4, False, 0.0), (2, True, 0.75))]


@pytest.mark.parametrize("dc,dv,slots,layered,alpha", CASES)
def test_irregular_rows_and_columns(dc, dv, slots, layered, alpha):
    rng = np.random.default_rng(100 * dc + 10 * dv + slots)
    m = 37
    h = irregular(rng, m, max(48, int(1.3 * m * (dc + 2) / 2 / dv) + dc), dc, dv)
    run(rng, h, slots, layered, alpha)


@pytest.mark.parametrize("max_iter", [40, 200])  # one- and two-byte flip words
@pytest.mark.parametrize("slots", [1, 2, 4, 8])
@pytest.mark.parametrize("m", [33, 64])
def test_regular_rows(m, slots, max_iter):
    rng = np.random.default_rng(m + slots)
    run(rng, regular(rng, m), slots, False, 0.625, max_iter, blocks=1)


# A lane per column: from one warp to the nineteen that a block holds (and one
# column more, which the teams serve), rows past the 128 of one residual look.
@pytest.mark.parametrize("m,alpha,max_iter", [(8, 0.625, 40), (16, 0.0, 40), (17, 0.625, 200), (48, 0.0, 200),
                                              (129, 0.625, 40), (304, 0.625, 30), (305, 0.625, 30)])
def test_column_path(m, alpha, max_iter):
    rng = np.random.default_rng(m)
    run(rng, regular(rng, m), 4, False, alpha, max_iter)


# The same for ten ones per row and five per column, at any batch size.
@pytest.mark.parametrize("m,alpha,max_iter", [(16, 0.625, 40), (17, 0.0, 200), (127, 0.0, 40), (304, 0.625, 130),
                                              (305, 0.625, 30)])
def test_column_path_ten_ones(m, alpha, max_iter):
    rng = np.random.default_rng(m)
    h = regular(rng, m, 10, 5)
    assert (h.sum(axis=0) == 5).all() and (h.sum(axis=1) == 10).all()
    run(rng, h, 1, False, alpha, max_iter)


# Lanes that loop over a long code's columns and rows: fewer, exactly as many and
# more of them than lanes; column degrees 0 to 3, row degrees 2 to 8.
@pytest.mark.parametrize("m,n,dc,alpha", [(480, 864, 8, 0.625), (432, 865, 8, 0.0), (700, 1800, 7, 0.625),
                                          (864, 1728, 8, 0.0)])
def test_long_codes(m, n, dc, alpha):
    rng = np.random.default_rng(m)
    h = irregular(rng, m, n, dc, 3)
    assert h.sum() > 2048
    run(rng, h, 1, False, alpha)


# Long codes of six ones per row and three per column: the lanes' loop up to
# 1.5e6 shots times columns (2192 shots here), teams beyond.
@pytest.mark.parametrize("alpha", [0.625, 0.0])
def test_long_exact_codes_by_batch(alpha):
    rng = np.random.default_rng(342)
    h = regular(rng, 342)
    m, n = h.shape
    idx = np.concatenate([np.nonzero(r)[0] for r in h])
    ptr = np.concatenate([[0], np.cumsum(h.sum(axis=1))])
    d = B.Decoder(ptr, idx, m, n, np.full(n, 0.03), B.Params(max_iter=40, alpha=alpha, w=4, short_iter=9))
    e = (rng.random((2193, n)) < 0.03).astype(np.uint8)
    synd = d.syndrome(torch.from_numpy(harness.pack_rows(e).view(np.int32)).cuda())
    few, many = d.decode(synd[:2192]), d.decode(synd)
    assert all(torch.equal(few[k], many[k][:2192]) for k in few)


@pytest.mark.parametrize("select", [B.BPSF_SELECT_MIN_WEIGHT, B.BPSF_SELECT_FIRST])
@pytest.mark.parametrize("shots", [1, 7, 8, 500])  # one and four slots per team
def test_column_path_equals_teams(shots, select):
    c = codes.bb("bb144")
    d = B.Decoder(c.ptr, c.idx, c.M, c.N, np.full(c.N, 0.07), B.Params(max_iter=60, w=6, short_iter=20, select=select))
    rng = np.random.default_rng(shots)
    e = (rng.random((shots, c.N)) < 0.08).astype(np.uint8)
    synd = d.syndrome(torch.from_numpy(harness.pack_rows(e).view(np.int32)).cuda())
    got = d.decode(synd)
    work = d.last_work()
    d.tuning = (1, 4, 8, 1, 1)  # blocks per SM given: the teams
    want = d.decode(synd)
    assert all(torch.equal(got[k], want[k]) for k in got)
    if select == B.BPSF_SELECT_MIN_WEIGHT:
        assert all(work[k] == v for k, v in d.last_work().items() if k != "slot_capacity")


@pytest.mark.parametrize("shots", [300, 20001])
def test_counters_outlive_the_workspace(shots):
    """A new trial list frees the workspace of a decode that may still be running."""
    c = codes.bb("bb144")
    d = B.Decoder(c.ptr, c.idx, c.M, c.N, np.full(c.N, 0.07), B.Params(max_iter=60, w=6, short_iter=20))
    rng = np.random.default_rng(shots)
    e = (rng.random((shots, c.N)) < 0.08).astype(np.uint8)
    synd = d.syndrome(torch.from_numpy(harness.pack_rows(e).view(np.int32)).cuda())
    d.decode(synd)
    want = d.last_work()
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    d.decode(synd, stream=stream, sync=False)
    d.set_trials([])
    B.bpsf_sync(d.handle, stream.cuda_stream)
    assert all(d.last_work()[k] == v for k, v in want.items() if k != "slot_capacity")


def run(rng, h, slots, layered, alpha, max_iter=40, blocks=0):
    m, n = h.shape
    idx = np.concatenate([np.nonzero(r)[0] for r in h])
    ptr = np.concatenate([[0], np.cumsum(h.sum(axis=1))])
    priors = rng.uniform(0.01, 0.2, n)
    P = B.Params(max_iter=max_iter, alpha=alpha, w=3, short_iter=9, layered=layered)
    d = B.Decoder(ptr, idx, m, n, priors, P)
    for warps in (1, 2):
        d.tuning = (warps, slots, 4, blocks, 1)
        shots = 301
        e = (rng.random((shots, n)) < priors).astype(np.uint8)
        s = (e.astype(np.int64) @ h.T.astype(np.int64) & 1).astype(np.uint8)
        s[::7] ^= (rng.random(s[::7].shape) < 0.5).astype(np.uint8)  # also syndromes that no run may satisfy
        oc = Code(h)
        op = OParams(P.max_iter, P.alpha, P.w, P.w_max, P.short_iter, P.select, layered=layered)
        eo, co, io, so = oc.bpsf_batch(s, priors, op, fp32=True, threads=THREADS)
        synd = torch.from_numpy(harness.pack_rows(s).view(np.int32)).cuda()
        g = {k: v.cpu().numpy() for k, v in d.decode_debug(synd).items()}
        assert (harness.unpack_rows(g["corr"].view(np.uint32), n) == eo).all()
        assert ((g["conv"] != 0) == co).all() and (g["iters"] == io).all() and (g["stage"] == so).all()
        plain = {k: v.cpu().numpy() for k, v in d.decode(synd).items()}
        assert all((plain[k] == g[k]).all() for k in plain)
        for i in range(0, shots, 43):
            r = oc.bp(s[i], priors, P.max_iter, P.alpha, track=True, layered=layered)
            assert (g["lout"][i] == np.asarray(r["lout"], dtype=np.float32)).all()
            assert (g["flips"][i] == r["flips"]).all()
