"""The hot pass's and the tail pass's candidate masks at their edges, event by
event against the oracle: plans of a few sub-steps, plans
that end inside, at and just past a window of 64 sub-steps, thresholds that
admit most sub-steps (large p_max) and almost none, and queues that hold one
particle per warp and many.  GPU only."""
import numpy as np
import pytest

import oracle as O
from paper_2008_10468_gb300 import inputs as I
from tests import parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


@pytest.mark.parametrize("p_max", [0.9, 0.2, 0.01, 0.0007])
@pytest.mark.parametrize("hot_min,tail_rows", [(1, 0), (1, 1 << 17), (64, 0)])
def test_plans_of_every_length_match_the_oracle(p_max, hot_min, tail_rows):
    arr = I.clumped_mixed(257, 31, hot_fraction=0.08, hot_chi=(0.5, 40.0))
    ctx = qed.Context(seed=17, p_max=p_max, dt=0.05)
    ctx.set_launch(hot_min=hot_min)
    ctx.set_tail(tail_rows)
    ctx.set_event_log(1 << 16)
    store = qed.ParticleStore.from_numpy(arr, capacity=40000)
    st = ctx.event_step(store, 4)
    ev, _ = ctx.read_event_log()
    cf = O.make_config(17, process_mask=3, cascade=1, p_max=p_max, dt=0.05)
    ost_store, ost, oev, oties = O.event_step(cf, arr, 4, capacity=40000)
    assert st["status"] == 0
    rep = parity.compare(ev, oev, oties, store.to_numpy(), ost_store, arr["id"])
    assert not rep["mismatches"], rep["mismatches"][:3]
    assert rep["exempt"] <= 1e-3 * rep["particles"] + 1
    if len(oties) == 0:
        for k in ("substeps", "emissions", "pairs", "children", "max_N"):
            assert st[k] == ost[k], (k, st[k], ost[k])


def test_full_grid_of_short_and_long_queues_agrees_with_the_thread_pass():
    # hot_min so large that the thread pass steps everything, against every
    # plan in the hot pass
    arr = I.clumped_mixed(70001, 33, hot_fraction=0.004)
    out = []
    for hot_min in (1, 1 << 20):
        ctx = qed.Context(seed=23)
        ctx.set_launch(hot_min=hot_min)
        ctx.set_tail(0)
        store = qed.ParticleStore.from_numpy(arr, capacity=300000)
        st = ctx.event_step(store, 9)
        a = store.to_numpy()
        o = np.argsort(a["id"], kind="stable")
        out.append((st, {k: v[o] for k, v in a.items()}))
    for k in ("substeps", "emissions", "pairs", "children", "plans", "candidates", "max_N"):
        assert out[0][0][k] == out[1][0][k], k
    for k in out[0][1]:
        np.testing.assert_array_equal(out[0][1][k], out[1][1][k])
