"""Performance cases: the decoding work that users of this library have it do.

Each case is one call (or one burst of requests) through the public entry
points of ``paper_2507_00254_gb300.bpsf``: batched decodes of one code, mixed
launches over several codes, host-buffer calls, the plain per-shot form, the
no-allocation form and the request server.  Codes, error rates, parameters and
launch shapes are those of the benchmark and the tests.

A case is a dict of plain values:
  form      batch | sync | multi | host | plain | noalloc | served
  codes     comma list of code names (one job per entry; one entry except for
            multi and served)
  p         comma list of physical error rates, one per entry
  shots     comma list of shot counts, one per entry (served: per code, split
            into requests)
  setting   decoder parameters, see SETTINGS
  first     first-success selection instead of minimum weight
  layered   layered schedule instead of flooding
  shape     launch shape W,S,B,blocks_per_sm,iter_chunk, or "" for the
            context's own
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_00254_gb300 import bpsf as B
from paper_2507_00254_gb300 import codes as C

# Decoder settings in use: the [[72]] example, the benchmark's code-capacity
# setting, the paper's code-capacity setting (adaptive damping, weight-1
# trials over |Phi| bits that depend on the code) and the phenomenological one.
SETTINGS = {
    "example": dict(max_iter=50, alpha=0.625, w=4, w_max=0, short_iter=10),
    "capacity": dict(max_iter=100, alpha=0.625, w=6, w_max=0, short_iter=20),
    "paper": dict(max_iter=50, alpha=0.0, w=None, w_max=1, short_iter=50),
    "phenom": dict(max_iter=200, alpha=0.625, w=5, w_max=0, short_iter=30),
}
PAPER_PHI = {"bb72": 4, "bb144": 7, "cbb126": 6, "gb254": 13, "cbb154": 8, "bb288": 20}
RANGES = {"example": (0.03, 0.06), "capacity": (0.02, 0.08), "paper": (0.04, 0.06), "phenom": (0.002, 0.004)}
NAMES = {"example": ("bb72",), "capacity": ("bb72", "bb90", "bb108", "bb144", "bb288"),
         "paper": ("bb72", "bb144", "cbb126", "gb254", "cbb154", "bb288"), "phenom": ("phenom144",)}
SIZE = {"bb72": (36, 72), "bb90": (45, 90), "bb108": (54, 108), "bb144": (72, 144), "bb288": (144, 288),
        "gb254": (127, 254), "cbb126": (63, 126), "cbb154": (77, 154), "phenom144": (864, 2592)}
EDGES = {n: 6 * m for n, (m, _) in SIZE.items()} | {"gb254": 1270, "phenom144": 6840}

# Mean BP iterations of one shot (trials included), as bpsf_last_work counts
# them, at the ends and inside of each setting's range of error rates.
MEAN_ITERS = {
    ("example", "bb72"): ((0.03, 6.3), (0.06, 36.2)),
    ("capacity", "bb72"): ((0.02, 8.0), (0.05, 110.0), (0.08, 346.0)),
    ("capacity", "bb90"): ((0.02, 6.6), (0.05, 165.0), (0.08, 609.0)),
    ("capacity", "bb108"): ((0.02, 6.3), (0.05, 161.0), (0.08, 656.0)),
    ("capacity", "bb144"): ((0.02, 5.5), (0.04, 61.6), (0.06, 302.0), (0.08, 695.0)),
    ("capacity", "bb288"): ((0.02, 8.6), (0.05, 144.0), (0.08, 847.0)),
    ("paper", "bb72"): ((0.04, 7.7), (0.06, 24.0)),
    ("paper", "bb144"): ((0.04, 13.3), (0.06, 71.6)),
    ("paper", "cbb126"): ((0.04, 11.4), (0.06, 56.6)),
    ("paper", "gb254"): ((0.04, 105.0), (0.06, 450.0)),
    ("paper", "cbb154"): ((0.04, 14.2), (0.06, 85.2)),
    ("paper", "bb288"): ((0.04, 28.8), (0.05, 84.5), (0.06, 204.0)),
    ("layered", "bb288"): ((0.04, 6.0), (0.05, 27.9), (0.06, 98.0)),
    ("phenom", "phenom144"): ((0.002, 1.6), (0.003, 2.6), (0.004, 4.3)),
}


def _case(name, form, codes, p, shots, setting, first=False, layered=False, shape=""):
    text = lambda v: ",".join("%g" % x if isinstance(x, float) else str(x) for x in v)  # noqa: E731
    return dict(name=name, form=form, codes=text(codes), p=text(p), shots=text(shots), setting=setting, first=first,
                layered=layered, shape=shape)


def listed():
    bb5 = ("bb72", "bb90", "bb108", "bb144", "bb288")
    return [
        # One syndrome of a quiet memory, waited for: a control loop's typical cycle.
        _case("one_shot", "sync", ["bb144"], [0.02], [1], "capacity"),
        # A handful of syndromes at a high rate, some of them failing: the tail of that loop
        # (100 iterations, then 63 trials of 20).
        _case("few_failing", "sync", ["bb144"], [0.08], [16], "capacity"),
        # The paper's own organisation: shot by shot, a launch for each run.
        _case("plain_64", "plain", ["bb144"], [0.04], [64], "capacity"),
        # The example workload: [[72,12,6]], 10^4 shots.
        _case("example_72", "batch", ["bb72"], [0.05], [10000], "example"),
        # A logical-error-rate point at a low rate: short runs, refills dominate.
        _case("low_rate_144", "batch", ["bb144"], [0.02], [100003], "capacity"),
        # Host buffers in and out, first valid trial wins: long runs and many trials.
        _case("host_first_144", "host", ["bb144"], [0.07], [60013], "capacity", first=True),
        # The headline workload at a quarter of its shots, at the shape the autotuner picks.
        _case("headline_144", "multi", ["bb144"] * 4, [0.02, 0.04, 0.06, 0.08], [250000] * 4, "capacity",
              shape="1,8,13,0,1"),
        # Five codes of uneven size and count in one launch.
        _case("mixed_five", "multi", bb5, [0.05] * 5, [60211, 13457, 88002, 41999, 25331], "capacity"),
        # Twelve rounds of noisy measurements, the largest matrix.
        _case("phenom_144", "batch", ["phenom144"], [0.004], [100000], "phenom"),
        # The paper's schedule for the [[288]] code.
        _case("layered_288", "batch", ["bb288"], [0.05], [100000], "paper", layered=True),
        # Rows of ten ones: the generalised bicycle code in the paper's setting.
        _case("paper_gb254", "batch", ["gb254"], [0.04], [50000], "paper"),
        # A burst of requests of six codes to the server.
        _case("served_mix", "served", bb5 + ("phenom144",), [0.05] * 5 + [0.003], [1200, 700, 900, 1500, 333, 401],
              "capacity", shape="1,1,15,0,1"),
    ]


def _setting(case, code):
    """A phenomenological code in a served mix keeps its own setting."""
    return "phenom" if code == "phenom144" else case["setting"]


def _lists(case):
    return (case["codes"].split(","), [float(x) for x in case["p"].split(",")],
            [int(x) for x in case["shots"].split(",")])


def _iters(case, code, p):
    """The layered schedule needs about a third of flooding's iterations."""
    key, scale = (_setting(case, code), code), 1.0
    if case["layered"]:
        key, scale = (("layered", code), 1.0) if ("layered", code) in MEAN_ITERS else (key, 1.0 / 3.0)
    pts = MEAN_ITERS[key]
    x = np.interp(p, [a for a, _ in pts], [math.log(b) for _, b in pts])
    return max(1.0, scale * math.exp(float(x)))


def _edge_updates(case):
    return sum(n * EDGES[c] * _iters(case, c, p) for c, p, n in zip(*_lists(case)))


def work(case):
    """bytes: packed syndromes in, corrections, flags, counts and stages out.  flops: per edge and
    iteration two comparisons for the two minima, one product and two sums."""
    names, _, shots = _lists(case)
    words = lambda b: 4 * ((b + 31) // 32)  # noqa: E731
    by = sum(n * (words(SIZE[c][0]) + words(SIZE[c][1]) + 4) for c, n in zip(names, shots))
    return {"bytes": by, "flops": 5.0 * _edge_updates(case)}


def draw(rng):
    """One more case: any form, code, option and launch shape of the ranges above."""
    most = max(_edge_updates(c) for c in listed())
    form = rng.choice(("batch", "batch", "batch", "sync", "multi", "multi", "host", "plain", "noalloc", "served"))
    setting = rng.choice(("capacity", "capacity", "paper", "example", "phenom"))
    if form == "served":
        setting = "capacity"
    lo, hi = RANGES[setting]
    names = NAMES[setting]
    if form == "multi":
        names = [rng.choice(names) for _ in range(rng.randint(2, 5))]
    elif form == "served":
        names = list(names) + ["phenom144"]
    else:
        names = [rng.choice(names)]
    top = {"sync": 64, "plain": 128, "noalloc": 32768, "served": 2000}.get(form, 200000)
    low = {"sync": 1, "plain": 4, "served": 100}.get(form, 300)
    p = [round(rng.uniform(*RANGES["phenom"]) if c == "phenom144" else rng.uniform(lo, hi), 4) for c in names]
    shots = [int(round(math.exp(rng.uniform(math.log(low), math.log(top))))) | 1 for _ in names]
    regular = all(c not in ("gb254", "phenom144") for c in names)
    case = _case("", form, names, p, shots, setting, first=rng.random() < 0.25,
                 layered=setting == "paper" and regular and rng.random() < 0.3,
                 shape=rng.choice(("", "", "1,4,12,0,1", "1,1,15,0,1", "2,2,14,0,1"))
                 if regular and form != "plain" else "")
    while _edge_updates(case) > most:
        shots = [max(1, n // 2) for n in shots]
        case["shots"] = ",".join(map(str, shots))
    del case["name"]
    return case


def _decoder(case, code, p):
    c = C.phenom("bb144") if code == "phenom144" else C.bb(code)
    setting = _setting(case, code)
    kw = dict(SETTINGS[setting])
    if kw["w"] is None:
        kw["w"] = PAPER_PHI[code]
    d = B.Decoder(c.ptr, c.idx, c.M, c.N, np.full(c.N, p), B.Params(
        select=B.BPSF_SELECT_FIRST if case["first"] else B.BPSF_SELECT_MIN_WEIGHT, layered=case["layered"], **kw))
    if case["shape"] and code != "phenom144":
        d.tuning = tuple(int(x) for x in case["shape"].split(","))
    return d


def _syndromes(dec, code, p, n, gen):
    """Packed syndromes of n random errors (measurement errors stop before the last, perfect round)."""
    rate = torch.full((dec.N,), p, device="cuda")
    if code == "phenom144":
        rate[-72:] = 0.0
    weight = (2 ** torch.arange(32, device="cuda", dtype=torch.int64))
    step = max(1, (1 << 25) // dec.N)
    out = []
    for a in range(0, n, step):
        m = min(step, n - a)
        bits = torch.zeros((m, 32 * dec.Wn), dtype=torch.int64, device="cuda")
        bits[:, :dec.N] = torch.rand((m, dec.N), device="cuda", generator=gen) < rate
        err = (bits.view(m, dec.Wn, 32) * weight).sum(2).to(torch.int32).contiguous()
        out.append(dec.syndrome(err))
    return torch.cat(out)


# A program keeps one server over its codes; it is kept here for the case that used it last.
_server = {"key": None, "decoders": None, "server": None}


def _served(case):
    key = repr(sorted((k, v) for k, v in case.items() if k not in ("name", "shots")))
    if _server["key"] != key:
        if _server["server"] is not None:
            _server["server"].stop()
        names, p, _ = _lists(case)
        _server["decoders"] = [_decoder(case, c, q) for c, q in zip(names, p)]
        _server["server"] = B.Server(_server["decoders"], max_inflight_shots=1 << 14)
        _server["key"] = key
    return _server["decoders"], _server["server"]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    names, p, shots = _lists(case)
    if case["form"] == "served":
        decs, server = _served(case)
    else:
        decs = [_decoder(case, c, q) for c, q in zip(names, p)]
    synds = [_syndromes(d, c, q, n, gen) for d, c, q, n in zip(decs, names, p, shots)]
    st = dict(form=case["form"], decs=decs, synds=synds)
    if case["form"] in ("batch", "multi", "plain", "noalloc"):
        st["outs"] = [d.outputs(n) for d, n in zip(decs, shots)]
    if case["form"] == "host":
        st["host"] = synds[0].cpu().numpy().view(np.uint32)
    if case["form"] == "served":
        # Requests of 1 to 256 shots, the codes interleaved.
        r = np.random.RandomState(seed % (1 << 32))
        requests = []
        for k, s in enumerate(synds):
            s, a = s.cpu().numpy().view(np.uint32), 0
            while a < s.shape[0]:
                b = min(s.shape[0], a + int(2 ** r.uniform(0, 8)))
                requests.append((k, a, s[a:b]))
                a = b
        order = sorted(range(len(requests)), key=lambda i: (requests[i][1] / shots[requests[i][0]], requests[i][0]))
        st.update(server=server, requests=[(requests[i][0], requests[i][2]) for i in order])
    return st


def run(st):
    form, decs, synds = st["form"], st["decs"], st["synds"]
    if form == "batch":
        return decs[0].decode(synds[0], out=st["outs"][0], sync=False)
    if form == "sync":
        return decs[0].decode(synds[0])
    if form == "multi":
        return B.decode_multi(decs, synds, outs=st["outs"], sync=False)
    if form == "host":
        return decs[0].decode_host(st["host"])
    if form == "plain":
        return decs[0].decode(synds[0], out=st["outs"][0], plain=True)
    if form == "noalloc":
        d, s, o = decs[0], synds[0], st["outs"][0]
        B.bpsf_decode_noalloc(d.handle, s.shape[0], s.data_ptr(), s.shape[1], o["corr"].data_ptr(), d.Wn,
                              o["conv"].data_ptr(), o["iters"].data_ptr(), o["stage"].data_ptr(),
                              torch.cuda.current_stream().cuda_stream)
        return o
    server = st["server"]
    tickets = [server.submit(k, s) for k, s in st["requests"]]
    parts = [[] for _ in decs]
    for t, (k, s) in zip(tickets, st["requests"]):
        parts[k].append(server.poll(t, s.shape[0], k))
    return [{key: np.concatenate([x[key] for x in v]) for key in v[0]} for v in parts]


def exact(case, seed):
    """Every output is a packed bit vector, a flag or a count: whole values, which stay the same."""
    return None
