"""A cascade step whose children are many times the store's free rows: the step
ends with QED_ERR_CAPACITY and a full store, writes nothing outside the store
and its own scratch, and leaves the context as good as new.  Only children whose
rows exist may enter the queue: parents go on emitting into a full store, so
the children asked for here (about nine an electron) are several times the
queue's entries.  GPU only."""
import ctypes as C

import numpy as np
import pytest

from paper_2008_10468_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402
from tests.test_zz_no_alloc import MAX_ROWS, _noalloc_fn, _noalloc_step  # noqa: E402

SEED = 31
FIELDS = tuple(qed.FLOAT_FIELDS) + ("id", "type")


def _sorted(a):
    o = np.argsort(a["id"], kind="stable")
    return {k: v[o] for k, v in a.items()}


def _cells(n):
    return (torch.arange(n, device="cuda") // 16).to(torch.int32), (n + 15) // 16


def _run(route, ctx, arr, cap, step, graph_steps=1):
    """(statistics of its steps, store) of one step by `route`."""
    n = len(arr["px"])
    if route == "host":
        store = qed.HostStore.from_numpy(arr, capacity=cap)
        return [ctx.event_step_host(store, step)], store
    store = qed.ParticleStore.from_numpy(arr, capacity=cap)
    if route == "graph":
        ctx.graph_capture(store, step, graph_steps)
        ctx.graph_launch()
        return ctx.graph_read_stats(), store
    if route == "cells":
        return [ctx.event_step_cells(store, step, *_cells(n))], store
    return [ctx.event_step(store, step)], store


@pytest.mark.parametrize("passes", [64, 63])
@pytest.mark.parametrize("route", ["step", "cells", "host", "graph"])
def test_overflow_stays_in_bounds(route, passes):
    n, cap, roomy = 2000, 2100, 2000 * 60
    arr = I.uniform_field_electrons(n, 20081047)
    ctx = qed.Context(seed=SEED, max_passes=passes)
    # neighbours: stores of the same size, allocated before and after the queue
    near = [qed.ParticleStore.from_numpy(arr, capacity=cap)]
    _run(route, ctx, arr, cap, 4, 2)
    near.append(qed.ParticleStore.from_numpy(arr, capacity=cap))
    before = [{k: getattr(s, k).clone() for k in FIELDS} for s in near]
    for k in range(4):
        st, store = _run(route, ctx, arr, cap, 5 + k, 2)
        assert st[0]["status"] == qed.QED_ERR_CAPACITY
        # more than the queue's 2 cap entries
        assert st[0]["required_capacity"] > 3 * cap
        if route == "host":
            assert store.count == n and st[0]["count"] == cap   # the host store is left as it was
        else:
            # full (a graph squeezes the decayed photons out after the step)
            assert store.n() == st[0]["count"] and n < store.n() <= cap
            assert store.n() == cap or route == "graph"
            ids = store.id[:n].cpu().numpy()
            np.testing.assert_array_equal(ids, np.asarray(arr["id"]).view(np.int64))
        if route == "graph":
            assert st[1]["status"] == qed.QED_ERR_CAPACITY and st[1]["substeps"] == 0
    for s, b in zip(near, before):
        for k in FIELDS:
            assert torch.equal(getattr(s, k), b[k]), k
    # few electrons in a store of that size next (entries of the overflowed steps
    # must be gone from the queue), then all in one with room: as in a fresh context
    few = {k: v[:40] for k, v in arr.items()}
    for a, c in ((few, cap), (arr, roomy)):
        ref = qed.Context(seed=SEED, max_passes=passes)
        sa, ga = _run(route, ref, a, c, 40)
        sb, gb = _run(route, ctx, a, c, 40)
        assert [s["status"] for s in sa] == [s["status"] for s in sb]
        assert sa[0]["status"] == 0
        for k in ("substeps", "emissions", "pairs", "children", "plans", "candidates", "count"):
            assert sa[0][k] == sb[0][k], k
        ga, gb = _sorted(ga.to_numpy()), _sorted(gb.to_numpy())
        for k in ga:
            np.testing.assert_array_equal(ga[k], gb[k], err_msg=k)


@pytest.mark.parametrize("n,cap", [(60000, MAX_ROWS), (2000, 2100)])
def test_noalloc_overflow_stays_in_bounds(n, cap):
    # 60000 electrons ask for about 5e5 children, four times the entries of the
    # built-in queue
    fn = _noalloc_fn()
    arr = I.uniform_field_electrons(n, 20081047)
    for k in range(3):
        status, st, got = _noalloc_step(fn, arr, cap, 5 + k, SEED)
        assert status == qed.QED_ERR_CAPACITY == st["status"]
        assert st["required_capacity"] > 3 * cap and st["count"] == cap == got.n()
        few = {f: v[:1500] for f, v in arr.items()}
        ref = qed.ParticleStore.from_numpy(few, capacity=MAX_ROWS)
        st_ref = qed.Context(seed=SEED).event_step(ref, 40 + k)
        status, st, got = _noalloc_step(fn, few, MAX_ROWS, 40 + k, SEED)
        assert status == qed.QED_OK == st_ref["status"]
        a, b = _sorted(ref.to_numpy()), _sorted(got.to_numpy())
        for f in a:
            np.testing.assert_array_equal(a[f], b[f], err_msg=f)


@pytest.mark.parametrize("n,seed", [(3000, 7), (70001, 8)])
def test_overflow_by_little(n, seed):
    # one row short, and the last pair of children split by the end of the store
    arr = I.clumped_mixed(n, 61, hot_fraction=0.05)
    full = qed.ParticleStore.from_numpy(arr, capacity=n * 30)
    total = qed.Context(seed=seed).event_step(full, 3)["count"]
    assert n < total < n * 30
    for short in (0, 1, 2, 3):
        ctx = qed.Context(seed=seed)
        store = qed.ParticleStore.from_numpy(arr, capacity=total - short)
        st = ctx.event_step(store, 3)
        assert st["count"] == store.n() == total - short
        assert st["status"] == (qed.QED_ERR_CAPACITY if short else 0)
        if short:
            assert total - short < st["required_capacity"] <= total
