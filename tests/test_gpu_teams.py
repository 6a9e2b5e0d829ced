"""One prior for all columns, on teams and on the column path.  Small launches
of exact-degree codes and long codes take the column path unless a number of
blocks per SM is given.  Both sides round every operation alike: results,
posteriors and flip counts equal those of the FP32 oracle, they are not close
to it."""
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
import synth  # noqa: E402
from oracle import Code, Params as OParams  # noqa: E402
from paper_2507_00254_gb300 import bpsf as B  # noqa: E402
from paper_2507_00254_gb300 import codes, harness  # noqa: E402

pytestmark = pytest.mark.gpu

THREADS = max(1, min(16, os.cpu_count() or 1))


class Workload:
    """Errors at one rate for all columns, and what the oracle makes of them."""

    def __init__(self, h, p, n, params, seed):
        self.h, self.p, self.P = h, p, params
        self.m, self.n = h.shape
        self.code = Code(h)
        self.s = self.code.syndrome(synth.bernoulli_bits(seed, 0, 0, n, self.n, p))
        self.want = self.code.bpsf_batch(self.s, p, self.oparams(), fp32=True, threads=THREADS)
        self.synd = torch.from_numpy(harness.pack_rows(self.s).view(np.int32)).cuda()
        idx = np.concatenate([np.nonzero(r)[0] for r in h])
        ptr = np.concatenate([[0], np.cumsum(h.sum(axis=1))])
        self.dec = B.Decoder(ptr, idx, self.m, self.n, np.full(self.n, p), params)

    def oparams(self):
        P = self.P
        return OParams(P.max_iter, P.alpha, P.w, P.w_max, P.short_iter, P.select, layered=P.layered)

    def check(self, out, shape):
        eo, co, io, so = self.want
        g = {k: v.cpu().numpy() for k, v in out.items()}
        assert (harness.unpack_rows(g["corr"].view(np.uint32), self.n) == eo).all(), shape
        assert ((g["conv"] != 0) == co).all() and (g["iters"] == io).all() and (g["stage"] == so).all(), shape

    def check_inside(self, shots):
        """Posteriors, flip counts and Phi of some initial runs."""
        g = {k: v.cpu().numpy() for k, v in self.dec.decode_debug(self.synd[:shots]).items()}
        for i in range(0, shots, 7):
            r = self.code.bp(self.s[i], self.p, self.P.max_iter, self.P.alpha, track=True, layered=self.P.layered)
            assert (g["lout"][i] == np.asarray(r["lout"], dtype=np.float32)).all()
            assert (g["flips"][i].astype(np.uint16) == r["flips"]).all()
            if not r["converged"]:
                assert (g["phi"][i] == oracle.top(r["flips"], self.P.w)).all()


def irregular(rng, m, n, dc, dv):
    """Row degrees 2..dc (at least one row of each end), column degrees at most dv."""
    h = np.zeros((m, n), dtype=np.uint8)
    for j in range(m):
        want = dc if j == 0 else (2 if j == 1 else int(rng.integers(2, dc + 1)))
        free = np.nonzero(h.sum(axis=0) < dv)[0]
        h[j, rng.choice(free, size=min(want, free.size), replace=False)] = 1
    return h


# With one prior and alpha = 1 or 1/2 all messages are one LLR times fractions of
# powers of two: sums cancel exactly, and zero messages of either sign meet zero
# sums.  A zero posterior is decided 1.
TIES = [("bb72", 0.06, 0.5), ("bb144", 0.07, 0.5), ("gb254", 0.04, 0.5), ((48, 72, 8, 4), 0.05, 1.0),
        ((60, 80, 16, 8), 0.05, 1.0), ((432, 865, 8, 3), 0.04, 1.0)]


@pytest.mark.parametrize("code,p,alpha", TIES, ids=str)
def test_zero_posteriors(code, p, alpha):
    h = codes.bb(code).dense() if isinstance(code, str) else irregular(np.random.default_rng(84), *code)
    w = Workload(h, p, 300 if h.sum() > 2048 else 1500, B.Params(max_iter=40, alpha=alpha, w=4, short_iter=15), 7100)
    shapes = [(1, 1, 2, 0), (1, 1, 2, 1), (1, 2, 4, 1)]
    if h.sum(axis=1).max() == 6:
        shapes += [(1, 4, 8, 1), (1, 8, 12, 1), (1, 8, 13, 1), (1, 2, 4, 2)]
    for shape in shapes:
        w.dec.tuning = shape
        w.check(w.dec.decode(w.synd), shape)
        w.check(w.dec.decode_debug(w.synd), shape)
    w.dec.tuning = (1, 1, 2, 0)
    whole = w.dec.decode(w.synd)
    for i in range(0, 300, 3):  # three at a time: one slot per team on the column path
        few = w.dec.decode(w.synd[i:i + 3])
        assert all(torch.equal(few[k], whole[k][i:i + 3]) for k in few)


_cache = {}


def workload(name, alpha, max_iter=100):
    """Two thousand shots of a code whose runs often fail; kept for the module."""
    key = (name, alpha, max_iter)
    if key not in _cache:
        p = {"bb72": 0.06, "bb144": 0.07, "gb254": 0.04}[name]
        P = B.Params(max_iter=max_iter, alpha=alpha, w=5, short_iter=20)
        w = Workload(codes.bb(name).dense(), p, 2000, P, 7100)
        assert (w.want[3] != 0).sum() > 10  # failed initial runs among them
        _cache[key] = w
    return _cache[key]


# (W, S, B, blocks per SM, iteration chunk).  One block per SM takes the
# full-register instance, two or more the 64-register one; thirteen teams of
# eight slots fit with one-byte flip words only.
TEAMS = [(1, 1, 4, 1), (1, 2, 15, 1), (1, 4, 15, 1), (1, 8, 12, 1), (1, 8, 13, 1), (1, 8, 13, 1, 2), (1, 16, 4, 1),
         (1, 32, 2, 1), (2, 2, 8, 1), (2, 8, 8, 1, 2), (4, 1, 12, 1, 3), (4, 16, 12, 1), (8, 1, 8, 1), (8, 32, 8, 1),
         (1, 32, 3, 1, 64), (1, 4, 15, 1, 8), (1, 4, 4, 2), (2, 2, 8, 2), (1, 1, 8, 2)]


@pytest.mark.parametrize("alpha", [0.625, 0.0])
@pytest.mark.parametrize("shape", TEAMS, ids=str)
def test_six_ones_per_row(shape, alpha):
    w = workload("bb144", alpha)
    w.dec.tuning = shape
    w.check(w.dec.decode(w.synd), shape)


@pytest.mark.parametrize("alpha", [0.625, 0.0])
@pytest.mark.parametrize("shape", [(1, 1, 4, 1), (1, 4, 12, 1), (1, 8, 12, 1), (1, 8, 13, 1), (2, 2, 8, 2)], ids=str)
def test_inside_six_ones_per_row(shape, alpha):
    w = workload("bb144", alpha)
    w.dec.tuning = shape
    w.check_inside(350)


def test_two_byte_flip_words():
    """More than 127 iterations: the shape for one-byte words is refused, the others count in two bytes."""
    w = workload("bb144", 0.625, 200)
    with pytest.raises(B.BpsfError):
        w.dec.tuning = (1, 8, 13, 1)
    for shape in ((1, 8, 12, 1), (1, 2, 4, 2)):
        w.dec.tuning = shape
        w.check(w.dec.decode(w.synd), shape)
        w.check_inside(100)


@pytest.mark.parametrize("alpha", [0.625, 0.0])
@pytest.mark.parametrize("shape", [(1, 1, 8, 1), (1, 2, 8, 1), (1, 4, 8, 1), (1, 8, 4, 1), (2, 16, 2, 1), (4, 2, 8, 2)],
                         ids=str)
def test_ten_ones_per_row(shape, alpha):
    w = workload("gb254", alpha)
    w.dec.tuning = shape
    w.check(w.dec.decode(w.synd), shape)
    w.check_inside(70)


# Row degrees 2 to dc, column degrees at most dv, one prior for all columns: the
# first iteration has no message set-up on teams, and one magnitude on the long
# codes' loop (the last two, where no blocks per SM are given).
@pytest.mark.parametrize("m,n,dc,dv", [(37, 60, 6, 3), (37, 60, 8, 4), (37, 80, 16, 8), (37, 90, 20, 16),
                                       (480, 864, 8, 3), (432, 865, 8, 3)])
@pytest.mark.parametrize("alpha", [0.625, 0.0])
def test_one_prior(m, n, dc, dv, alpha):
    h = irregular(np.random.default_rng(1000 * dc + n), m, n, dc, dv)
    w = Workload(h, 0.04, 300, B.Params(max_iter=40, alpha=alpha, w=3, short_iter=9), 7200 + n)
    for shape in ((1, 1, 2, 1), (1, 2, 4, 1), (2, 4, 4, 1), (2, 2, 4, 0)):
        if m > 100 and shape[1] > 2:
            continue  # no room for four slots of a long code in two teams
        w.dec.tuning = shape
        w.check(w.dec.decode(w.synd), shape)
        w.check_inside(70)


def test_uneven_codes_in_one_launch():
    """Exact codes beside the phenomenological one: the instance with both team loops."""
    P = B.Params(max_iter=100, alpha=0.0, w=5, short_iter=20)
    works = [workload("bb72", 0.0), Workload(codes.phenom("bb144").dense(), 0.004, 1200, P, 7300), workload("bb144", 0.0)]
    for w, shape in zip(works, ((1, 2, 4, 1), (2, 1, 4, 1), (1, 4, 4, 1))):
        w.dec.tuning = shape
    for w, out in zip(works, B.decode_multi([w.dec for w in works], [w.synd for w in works])):
        w.check(out, "mixed")


def test_plain_form_takes_the_given_shape():
    """Blocks per SM given: the initial runs of the plain form are teams of one slot.  (With
    4095 trials the column path would hold four slots, three of them idle.)"""
    P = B.Params(max_iter=60, alpha=0.625, w=12, short_iter=3)
    w = Workload(codes.bb("bb144").dense(), 0.02, 40, P, 7400)
    conv = np.nonzero(w.want[3] == 0)[0]
    assert conv.size > 20
    for shape in ((1, 4, 8, 1), (2, 2, 4, 2)):
        w.dec.tuning = shape
        out = w.dec.decode(w.synd[torch.from_numpy(conv).cuda()].contiguous(), plain=True, sync=False)
        assert (out["iters"].cpu().numpy() == w.want[2][conv]).all() and (out["stage"] == 0).all()
        work = w.dec.last_work()
        assert work["iterations"] == w.want[2][conv].sum() and work["slot_capacity"] == work["iterations"]
        w.check(w.dec.decode(w.synd, plain=True), shape)


def test_plain_form_runs_one_shot_on_one_slot():
    """However many trials a code has, an initial run of the plain form leaves no slot idle."""
    P = B.Params(max_iter=60, alpha=0.625, w=12, short_iter=3)
    w = Workload(codes.bb("bb144").dense(), 0.02, 40, P, 7400)
    synd = w.synd[torch.from_numpy(np.nonzero(w.want[3] == 0)[0]).cuda()].contiguous()
    w.dec.decode(synd, plain=True, sync=False)
    work = w.dec.last_work()
    assert work["iterations"] > 0 and work["slot_capacity"] == work["iterations"]


@pytest.mark.parametrize("code,p,shots", [("gb254", 0.04, 4000), ((432, 865, 8, 3), 0.02, 1000)], ids=str)
def test_autotuned_shape_is_the_one_that_decodes(code, p, shots):
    """Codes with a shape of their own at any batch size: the autotuner leaves it, or sets a
    faster team shape with its blocks per SM."""
    h = codes.bb(code).dense() if isinstance(code, str) else irregular(np.random.default_rng(84), *code)
    w = Workload(h, p, 300, B.Params(max_iter=30, alpha=0.625, w=2, short_iter=9), 7500)
    before = w.dec.tuning
    chosen = w.dec.autotune(p_sample=p, n_sample=shots)
    assert w.dec.tuning == chosen and (chosen == before or chosen[3] > 0)
    assert before[3] == 0
    w.check(w.dec.decode(w.synd), chosen)
