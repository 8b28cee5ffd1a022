"""The push step's candidate windows at their edges, event by event against the
oracle: plans of a few sub-steps and plans that end inside, at and past a window
of 64, thresholds that admit most sub-steps (large p_max) and almost none, one
row, a few and more than one warp takes, and emission alone.  GPU only."""
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


@pytest.mark.parametrize("n", [1, 33, 300])
@pytest.mark.parametrize("p_max,dt", [(0.9, 0.02), (0.2, 0.02), (0.01, 0.02), (0.002, 0.005)])
@pytest.mark.parametrize("cascade", [0, 1])
def test_push_plans_of_every_length_match_the_oracle(n, p_max, dt, cascade):
    arr = I.clumped_mixed(n, 41, hot_fraction=0.1, hot_chi=(0.5, 40.0))
    cap = 64 * n + 4000
    ctx = qed.Context(seed=19, p_max=p_max, dt=dt, cascade=bool(cascade))
    ctx.set_event_log(1 << 16)
    store = qed.ParticleStore.from_numpy(arr, capacity=cap)
    st = ctx.event_step(store, 2, push=True)
    ev, _ = ctx.read_event_log()
    cf = O.make_config(19, process_mask=3, cascade=cascade, p_max=p_max, dt=dt, push=1)
    ost_store, ost, oev, oties = O.event_step(cf, arr, 2, capacity=cap)
    assert st["status"] == 0
    rep = parity.compare(ev, oev, oties, store.to_numpy(), ost_store, arr["id"])
    assert not rep["mismatches"], rep["mismatches"][:3]
    assert rep["exempt"] <= 1e-3 * rep["particles"] + 1
    if len(oties) == 0:
        for k in ("substeps", "emissions", "pairs", "children", "plans", "max_N"):
            assert st[k] == ost[k], (k, st[k], ost[k])
