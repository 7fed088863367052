"""Every binding that hands pointers to the library refuses arrays that are too short, before the library is called.

The C entry points take no lengths, so a short array (a state of another
level, a hierarchy's maps in the order the coarsening made them) would be read
or written past its end on the device.  Nothing here needs a GPU: the library
is replaced by one that fails the test when it is reached.
"""
from types import SimpleNamespace

import numpy as np
import pytest

from paper_2504_12013_gb300 import jet, synth

torch = pytest.importorskip("torch")

K = 4


class _Unreachable:
    def __getattr__(self, name):
        raise AssertionError(f"{name} was reached with a short array")


@pytest.fixture(autouse=True)
def no_library(monkeypatch):
    monkeypatch.setattr(jet, "load_library", _Unreachable)
    monkeypatch.setattr(jet, "_ptr", lambda t, dtype=None, name="tensor": None if t is None else t.data_ptr())
    monkeypatch.setattr(jet, "_stream_ptr", lambda stream: None)


def ctx(n, m):
    return jet.Ctx(None, SimpleNamespace(n=n, m=m), jet.params(K))


def ints(count, dtype=torch.int32):
    return torch.zeros(count, dtype=dtype)


def state(n, m, k=K):
    return SimpleNamespace(part=ints(n), phi=ints(m * k), block_w=ints(k, torch.int64))


def cut(t):
    return t[:-1]


def short_calls():
    """(name, call): each call has one array that is one entry short."""
    c, n, m = ctx(10, 6), 10, 6
    full = dict(part=ints(n), phi=ints(m * K), block_w=ints(K, torch.int64), locked=ints(n, torch.uint8),
                stats=ints(8, torch.int64), target=ints(n), gain=ints(n), in_m=ints(n, torch.uint8), rg=ints(n),
                approved=ints(n, torch.uint8), objective_out=ints(1, torch.int64))
    takes = {"jet_build_pincounts": ("part", "phi", "block_w"), "jet_connectivity": ("phi", "objective_out"),
             "jet_refine_round": ("part", "phi", "block_w", "locked", "stats"),
             "jet_rebalance": ("part", "phi", "block_w", "stats"), "jet_refine": ("part", "phi", "block_w"),
             "jet_candidates": ("part", "phi", "locked", "target", "gain", "in_m"),
             "jet_afterburner": ("part", "phi", "rg", "approved"), "jet_quotient_schedule": ("phi",)}
    first = {"jet_refine_round": ((3, 4),), "jet_candidates": ((3, 4),), "jet_refine": (((3, 4),), 8)}
    for f, names in takes.items():
        for bad in names:
            args = [cut(full[x]) if x == bad else full[x] for x in names]
            yield f"{f}-{bad}", lambda f=f, args=args: getattr(jet, f)(c, *first.get(f, ()), *args)
    levels = [ctx(5, 3), ctx(10, 6), ctx(20, 12)]
    states = [state(5, 3), state(10, 6), state(20, 12)]
    yield "uncoarsen-maps-finest-first", lambda: jet.jet_uncoarsen(levels, [ints(20), ints(10)], (), 8, states)
    yield "uncoarsen-map", lambda: jet.jet_uncoarsen(levels, [ints(10), ints(19)], (), 8, states)
    yield "uncoarsen-states-finest-first", lambda: jet.jet_uncoarsen(levels, [ints(10), ints(20)], (), 8, states[::-1])
    yield "uncoarsen-few-states", lambda: jet.jet_uncoarsen(levels, [ints(10), ints(20)], (), 8, states[:2])
    batch = jet.Batch(None, levels)
    for f, more in (("jet_batch_refine", ()), ("jet_batch_tune", ([0],)), ("jet_batch_autotune", ([(1, 256)],))):
        for what, st in (("order", states[::-1]), ("few", states[:2]),
                         ("phi", [*states[:2], SimpleNamespace(**{**vars(states[2]), "phi": ints(12 * K - 1)})])):
            yield f"{f}-{what}", lambda f=f, st=st, more=more: getattr(jet, f)(batch, (), 8, st, *more)
    dev = {"eptr": ints(m + 1, torch.int64), "pins": ints(12), "vptr": ints(n + 1, torch.int64), "inc": ints(12),
           "vwgt": ints(n), "ewgt": ints(m)}
    dh = jet.DeviceHypergraph.from_tensors(n, m, 12, **dev)
    for bad in dev:
        yield f"hypergraph-{bad}", lambda bad=bad: jet.DeviceHypergraph.from_tensors(
            n, m, 12, **{**dev, bad: cut(dev[bad])}).c()
    yield "cluster-order", lambda: jet.jet_cluster(dh, 5, ints(n - 1))
    yield "contract-label", lambda: jet.jet_contract(dh, ints(n - 1))
    yield "noalloc-vwgt", lambda: jet.jet_block_weights_noalloc(ints(n), ints(n - 1), K, ints(K, torch.int64))
    yield "noalloc-block_w", lambda: jet.jet_block_weights_noalloc(ints(n), ints(n), K, ints(K - 1, torch.int64))
    h = synth.from_edges(4, [[0, 1], [1, 2, 3]])
    part = np.zeros(4, np.int32)
    for bad in ("eptr", "pins", "vptr", "inc", "vwgt", "ewgt"):
        short = SimpleNamespace(n=h.n, m=h.m, P=h.P, **{x: getattr(h, x)[: len(getattr(h, x)) - (x == bad)] for x in
                                                       ("eptr", "pins", "vptr", "inc", "vwgt", "ewgt")})
        yield f"refine_host-{bad}", lambda short=short: jet.jet_refine_host(short, jet.params(2), (), 8, part)
        yield f"submit-{bad}", lambda short=short: jet.jet_server_submit(SimpleNamespace(handle=1, keep={}), short,
                                                                         jet.params(2), (), 8, part)
    yield "refine_host-part", lambda: jet.jet_refine_host(h, jet.params(2), (), 8, part[:3].copy())
    yield "rounds_host-part", lambda: jet.jet_rounds_host(h, jet.params(2), (3, 4), 1, part[:3].copy())


@pytest.mark.parametrize("name", [n for n, _ in short_calls()])
def test_short_array_is_refused(name):
    with pytest.raises(ValueError, match="at least|states for"):
        dict(short_calls())[name]()


def test_full_arrays_reach_the_library():
    levels, states = [ctx(5, 3), ctx(10, 6)], [state(5, 3), state(10, 6)]
    with pytest.raises(AssertionError, match="jet_uncoarsen was reached"):
        jet.jet_uncoarsen(levels, [ints(10)], (), 8, states)
    c = ctx(10, 6)
    c.graph_path = True  # phi is not touched there: a placeholder stays accepted
    with pytest.raises(AssertionError, match="jet_refine_round was reached"):
        jet.jet_refine_round(c, (3, 4), ints(10), ints(1), ints(K, torch.int64), ints(10, torch.uint8))
