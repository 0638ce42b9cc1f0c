"""The walks with producers against the per-event, windowed and staged walks, bit for bit.

Which walk a call takes follows from the pool and the number of streams, so streams without
events beside the same real ones bring the same call onto the other walk: more than 1,536
streams for the windowed walk of pools of at most 16 decodes, more than 512 Ki decodes over all
streams for the staged walk of 513 .. 1,024 decodes, more than 256 Ki for the per-event walks of
self-contention and the load model (pools above 96), and more streams an SM than the rule allows
(walk_pays) for the packed per-event walks of small pools and the others.  Fewer such streams keep
the walk and narrow its CTAs (64 and 128 threads, shorter windows), which are compared too.  Pools
of 17 .. 512 decodes with base scores
are compared with self-contention at counter cap 0 with its workspace, the same greedy on the
per-event walk.  The event lists are those of tests/test_gpu_window.py: departures in the same
window, the next, later or never, twice, requests renumbered at random, 2^27 tokens and more,
bad events, initial loads.  What has no second walk (self-contention, 17 .. 32 decodes) is held
against the oracle at the edges of the pool sizes and of the counters kept in registers (32
prefill ranks)."""
import numpy as np
import pytest

import synth
from tests.gpu_common import THETA
from tests.test_gpu_inflight import test_inflight_streams_vs_oracle as inflight_vs_oracle
from tests.test_gpu_load import T_A, T_B, test_load_streams_vs_oracle as load_vs_oracle
from tests.test_gpu_window import _case, _renumber, _run

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()


def nk():
    from paper_2606_03910_gb300 import netkv
    return netkv


def _arrays(c, twice):
    a = dict(length=c["length"], prefill=c["prefill"], snap=c["snap"],
             arrival_us=c["arrival_us"], events=c["events"], M=c["M"])
    if twice:  # the first stream's last departure again, and one of them early
        e0, e1 = int(c["event_off"][0]), int(c["event_off"][1])
        ev = a["events"].copy()
        dep = np.flatnonzero(ev[e0:e1] >> 31) + e0
        ev[dep[-1]] = ev[dep[-2]]
        ev[dep[5]] = ev[dep[4]]
        a["events"] = ev
    return a


def _call(c, a, form, pad, load_init=None, model=None, cap=4, bpt=synth.BYTES_PER_TOKEN_SHARD,
          back=False):
    """The greedy `form` with `pad` streams without events after the real ones; the results
    of the real streams.  back: the last stream's offsets run back to 0."""
    netkv = nk()
    from paper_2606_03910_gb300.pipeline import weights_tensor
    sc, x, out = c["sc"], c["x"], c["out"]
    R, D, S = x.R, sc.D, x.n_streams + pad
    t32 = lambda v: torch.from_numpy(np.asarray(v).astype(np.uint32).view(np.int32)).cuda()
    off = np.concatenate([c["event_off"], np.full(pad, c["event_off"][-1], np.int64)])
    if back:
        off[-1] = 0
    wt = weights_tensor(np.concatenate([c["w"].weights, np.repeat(c["w"].weights[:1], pad, 0)]),
                        THETA, c["cap"], bpt)
    init = None
    if load_init is not None:
        init = torch.zeros((S, D), dtype=torch.int64, device="cuda")
        init[:x.n_streams] = load_init
    f = lambda *shape, dtype: torch.full(shape, -9, dtype=dtype, device="cuda")
    o = dict(dec=f(R, dtype=torch.int32), best=f(R, dtype=torch.float32),
             second=f(R, dtype=torch.float32), load=f(S, D, dtype=torch.int64),
             status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    head = (sc.topo, S, wt)
    req = (R, t32(a["length"]), t32(a["prefill"]), t32(a["snap"]))
    ev = (x.n_snap, t32(a["events"]), torch.from_numpy(off).cuda())
    if form == "plain":
        ws = torch.empty(netkv.netkv_schedule_workspace_size(R, D), dtype=torch.uint8, device="cuda")
        netkv.netkv_schedule_streams(*head, *req, a["M"], out.UB, *ev, init, o["dec"], o["best"],
                                     o["second"], o["load"], o["status"], workspace=ws)
    elif form == "inflight":
        o["xfer"] = f(R, dtype=torch.int32)
        netkv.netkv_schedule_streams_inflight(*head, *req, torch.from_numpy(a["arrival_us"]).cuda(),
                                              a["M"], out.UB, *ev, cap, init, o["dec"], o["best"],
                                              o["second"], o["xfer"], o["load"], o["status"])
    else:
        o["n"] = f(S, D, dtype=torch.int32)
        n_init = None if init is None else (init.abs() % 7).to(torch.int32)
        netkv.netkv_schedule_streams_load(*head, netkv.LoadModel(T_A, T_B, *model), *req, a["M"],
                                          out.UB, *ev, init, n_init, o["dec"], o["best"],
                                          o["second"], o["load"], o["n"], o["status"])
    torch.cuda.synchronize()
    if back:  # the stream has no events: its loads are the initial ones
        assert (o["load"][-1] == (model[3] if form == "load" and init is None else 0)).all()
    for k in ("load", "n"):
        if k in o:
            o[k] = o[k][:x.n_streams]
    return o


def _same(a, b):
    for k in a:
        assert torch.equal(a[k], b[k]), k
    assert (a["dec"] >= 0).any()


def _init(c, seed=3):
    rng = np.random.default_rng(seed)
    return torch.from_numpy(rng.integers(-50, 30_000, (c["x"].n_streams, c["sc"].D))).cuda()


KINDS = ["plain", "huge", "bad", "load_init", "twice"]


@pytest.mark.parametrize("fanout,D,pad", [((1, 1, 1, 2), 1, 1540),     # one decode
                                          ((1, 2, 3, 5), 15, 1540),    # against 16-lane segments
                                          ((2, 2, 2, 4), 16, 1540),
                                          ((1, 1, 577, 2), 577, 920),  # against the staged walk
                                          ((2, 8, 16, 8), 1024, 520)])
@pytest.mark.parametrize("kind", KINDS)
def test_base_scores_with_and_without_more_streams(fanout, D, pad, kind):
    c = _case(fanout, 3, rps=150, seed=D, huge=kind == "huge", bad=kind == "bad")
    assert c["sc"].D == D
    init = _init(c) if kind == "load_init" else None
    a = _arrays(c, kind == "twice")
    _same(_call(c, a, "plain", 0, init), _call(c, a, "plain", pad, init))


@pytest.mark.parametrize("fanout,D", [((1, 1, 17, 2), 17), ((1, 1, 31, 2), 31), ((2, 2, 4, 4), 32),
                                      ((1, 1, 33, 2), 33), ((1, 1, 65, 2), 65),
                                      ((1, 2, 49, 2), 98), ((2, 4, 8, 9), 288)])
@pytest.mark.parametrize("kind", KINDS)
def test_base_scores_against_the_per_event_walk(fanout, D, kind):
    c = _case(fanout, 3, rps=150, seed=D, huge=kind == "huge", bad=kind == "bad")
    assert c["sc"].D == D
    init = _init(c) if kind == "load_init" else None
    for a in (_arrays(c, kind == "twice"), _renumber(c)):
        ref = _run(c, a, "packed", init)
        got = _run(c, a, "window", init)  # the form with base scores
        _same(got, ref)


@pytest.mark.parametrize("fanout,D,pad", [((1, 1, 97, 2), 97, 2800), ((2, 4, 8, 9), 288, 920)])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("cap", [0, 1, 255])
def test_self_contention_with_and_without_more_streams(fanout, D, pad, kind, cap):
    c = _case(fanout, 2, rps=150, seed=D, huge=kind == "huge", bad=kind == "bad")
    assert c["sc"].D == D
    init = _init(c) if kind == "load_init" else None
    c["prefill"][c["prefill"] < c["sc"].P] %= 3           # many transfers of one prefill
    c["arrival_us"] = c["arrival_us"] // 50               # more pending than a warp's lanes
    a = _arrays(c, kind == "twice")
    _same(_call(c, a, "inflight", 0, init, cap=cap), _call(c, a, "inflight", pad, init, cap=cap))


@pytest.mark.parametrize("fanout,D,pad", [((1, 1, 97, 2), 97, 2800), ((2, 4, 8, 9), 288, 920)])
@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("model,bpt", [((4, 0, 10 ** 8, 3 * 10 ** 9), synth.BYTES_PER_TOKEN_SHARD),
                                       ((64, 0, 0, 10 ** 12), 0),
                                       ((2, 0, 0, 1 << 60), (1 << 31) + 7)])
def test_load_model_with_and_without_more_streams(fanout, D, pad, kind, model, bpt):
    c = _case(fanout, 2, rps=150, seed=D, huge=kind == "huge", bad=kind == "bad")
    assert c["sc"].D == D
    init = _init(c) + model[3] if kind == "load_init" else None
    a = _arrays(c, kind == "twice")
    kw = dict(load_init=init, model=model, bpt=bpt)
    _same(_call(c, a, "load", 0, **kw), _call(c, a, "load", pad, **kw))


@pytest.mark.parametrize("fanout,D", [((1, 1, 31, 2), 31), ((2, 2, 4, 4), 32),
                                      ((1, 1, 13, 5), 32),   # 33 prefill ranks
                                      ((1, 1, 33, 2), 33), ((1, 2, 24, 4), 96)])
def test_small_pools_against_the_oracle(fanout, D):
    inflight_vs_oracle(fanout, "alternate", D, 2, False)
    load_vs_oracle(fanout, "alternate", D, 4, 10 ** 8, 6 * 10 ** 8)


@pytest.mark.parametrize("fanout,D,pad", [((2, 2, 2, 2), 8, 1100), ((2, 2, 2, 4), 16, 1100),
                                          ((2, 2, 2, 2), 8, 1540), ((2, 2, 2, 4), 16, 1540),
                                          ((2, 2, 4, 4), 32, 1100), ((2, 4, 8, 9), 288, 1100),
                                          ((2, 8, 16, 8), 1024, 520), ((1, 1, 1025, 2), 1025, 2)])
@pytest.mark.parametrize("form", ["plain", "inflight", "load"])
def test_offsets_that_decrease(fanout, D, pad, form):
    """A stream whose event offsets decrease has no events, in the base-score pass as in the
    walk; the other streams' results are those of a call without it."""
    c = _case(fanout, 3, rps=150, seed=D)
    assert c["sc"].D == D
    a = _arrays(c, False)
    kw = dict(model=(4, 0, 10 ** 8, 3 * 10 ** 9)) if form == "load" else {}
    _same(_call(c, a, form, 0, **kw), _call(c, a, form, pad, back=True, **kw))


@pytest.mark.parametrize("fanout,D,form,pad", [
    ((2, 2, 2, 2), 8, "plain", 0), ((2, 2, 2, 2), 8, "plain", 1540), ((2, 2, 2, 4), 16, "plain", 1540),
    ((2, 4, 8, 9), 288, "plain", 0), ((2, 8, 16, 8), 1024, "plain", 520),
    ((1, 1, 1025, 2), 1025, "plain", 0), ((2, 2, 2, 2), 8, "inflight", 0),
    ((2, 4, 8, 9), 288, "inflight", 0), ((2, 2, 2, 2), 8, "load", 0), ((2, 4, 8, 9), 288, "load", 0),
    ((2, 4, 8, 9), 288, "load", 920)])
def test_event_code_of_all_ones(fanout, D, form, pad):
    """0xffffffff is the departure of an out-of-range request: skipped, and flagged as such."""
    c = _case(fanout, 3, rps=150, seed=D)
    a = _arrays(c, False)
    kw = dict(model=(4, 0, 10 ** 8, 3 * 10 ** 9)) if form == "load" else {}
    at = np.flatnonzero(a["events"] >> 31)[40]
    got = []
    for code in (0xffffffff, (c["x"].R + 7) | 0x80000000):
        ev = a["events"].copy()
        ev[at] = code
        got.append(_call(c, dict(a, events=ev), form, pad, **kw))
    _same(*got)
    assert int(got[0]["status"].item()) == nk().NETKV_DEV_ERANGE


@pytest.mark.parametrize("fanout,D,form,pad", [
    ((2, 2, 2, 2), 8, "plain", 0), ((2, 4, 8, 9), 288, "plain", 0), ((2, 8, 16, 8), 1024, "plain", 520),
    ((1, 1, 1025, 2), 1025, "plain", 0), ((2, 2, 2, 2), 8, "inflight", 0),
    ((2, 4, 8, 9), 288, "inflight", 0), ((2, 4, 8, 9), 288, "inflight", 920)])
def test_no_token_limit_and_negative_loads(fanout, D, form, pad):
    """A capacity of 2^63 - 1 tokens limits nothing, also where loads are negative (departures
    of requests that an earlier call dispatched)."""
    c = _case(fanout, 2, rps=150, seed=D)
    a = _arrays(c, False)
    init = _init(c) - 40_000
    got = []
    for cap in (2 ** 63 - 1, 2 ** 62):
        got.append(_call(dict(c, cap=cap), a, form, pad, init))
    _same(*got)


@pytest.mark.parametrize("fanout,D,pad", [((2, 2, 2, 2), 8, 0), ((2, 4, 8, 9), 288, 0),
                                          ((2, 4, 8, 9), 288, 920)])
def test_load_model_with_memory_near_its_range(fanout, D, pad):
    """Free memory up to 2^63 - 1 bytes, a token of one byte, and a reserve of 2^62 bytes."""
    c = _case(fanout, 2, rps=150, seed=D)
    a = _arrays(c, False)
    call = lambda m_min, m0, bpt: _call(c, a, "load", pad, model=(64, 0, m_min, m0), bpt=bpt)
    for other, shift, bpt in (((0, 2 ** 63 - 1), 2 ** 62 - 1, 1),
                              ((2 ** 62, 2 ** 62 + 2 * 10 ** 8), 0, synth.BYTES_PER_TOKEN_SHARD)):
        base = (0, 2 ** 62) if bpt == 1 else (0, 2 * 10 ** 8)
        x, y = call(*other, bpt), call(*base, bpt)
        x["load"] -= other[1] - base[1]
        _same(x, y)


# streams without events beside two real ones, at 152 SMs: (pool, streams, whether the walk stays)
FLEETS = {
    "inflight": [((1, 1, 3, 2), 3, 700), ((2, 2, 2, 2), 8, 700), ((2, 2, 2, 4), 16, 700),
                 ((1, 1, 24, 2), 24, 700), ((2, 2, 4, 4), 32, 1300), ((1, 1, 13, 5), 32, 700),
                 ((1, 1, 33, 2), 33, 400), ((1, 1, 33, 2), 33, 1300), ((1, 1, 64, 2), 64, 700),
                 ((1, 1, 96, 2), 96, 400), ((1, 1, 97, 2), 97, 280),
                 # past the rule: the per-event walks
                 ((1, 1, 3, 2), 3, 4300), ((2, 2, 2, 2), 8, 4300), ((2, 2, 2, 4), 16, 3100),
                 ((1, 1, 65, 2), 65, 700), ((1, 1, 129, 2), 129, 400)],
    "load": [((1, 1, 3, 2), 3, 700), ((2, 2, 2, 2), 8, 1300), ((2, 2, 2, 4), 16, 700),
             ((2, 2, 4, 4), 32, 700), ((1, 1, 33, 2), 33, 400), ((1, 1, 65, 2), 65, 1300),
             ((1, 1, 96, 2), 96, 700), ((1, 1, 97, 2), 97, 400), ((2, 4, 8, 9), 288, 400),
             ((1, 1, 3, 2), 3, 4900), ((2, 2, 2, 4), 16, 2500), ((2, 2, 4, 4), 32, 1300),
             ((1, 1, 130, 2), 130, 700), ((1, 1, 401, 2), 401, 320)],
    "plain": [((2, 2, 2, 2), 8, 700), ((2, 2, 4, 4), 32, 1300), ((1, 1, 33, 2), 33, 400),
              ((1, 1, 65, 2), 65, 1300), ((2, 4, 8, 9), 288, 400), ((2, 4, 8, 9), 288, 1300),
              ((1, 1, 513, 2), 513, 400), ((1, 1, 513, 2), 513, 650), ((1, 1, 801, 2), 801, 320)],
}


@pytest.mark.parametrize("form,fanout,D,pad", [(f, *v) for f in FLEETS for v in FLEETS[f]])
@pytest.mark.parametrize("kind", ["plain", "bad", "load_init", "twice"])
def test_fleets(form, fanout, D, pad, kind):
    c = _case(fanout, 2, rps=150, seed=D, bad=kind == "bad")
    assert c["sc"].D == D
    model = (4, 0, 10 ** 8, 3 * 10 ** 9)
    init = _init(c) + (model[3] if form == "load" else 0) if kind == "load_init" else None
    if form == "inflight":
        c["prefill"][c["prefill"] < c["sc"].P] %= 40
        c["arrival_us"] = c["arrival_us"] // 50
    a = _arrays(c, kind == "twice")
    kw = dict(load_init=init, **(dict(model=model) if form == "load" else {}))
    _same(_call(c, a, form, 0, **kw), _call(c, a, form, pad, **kw))
