"""The bounded wait of the persistent cascade pass counts from the last progress
of the step: with a limit far below the step's length (and far above the gaps
between two events anywhere) no warp may give up, however long it has idled
before it takes an entry that is still being written.  A handful of electrons in
a long step: most warps idle for most of it, and entries come one by one.  GPU
only."""
import pytest

from paper_2008_10468_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


@pytest.mark.parametrize("n,dt", [(20, 3.0), (400, 0.5)])
def test_idle_warps_that_take_an_entry_do_not_time_out(n, dt):
    # steps of 4 to 25 ms, a limit of 0.3 ms
    arr = I.uniform_field_electrons(n, 20081047)
    keys = ("status", "substeps", "emissions", "pairs", "children", "plans", "count")
    for k in range(8):
        st = []
        for limit in (0, 300000):
            ctx = qed.Context(seed=100 + k, dt=dt)
            ctx.set_wait_limit(limit)
            store = qed.ParticleStore.from_numpy(arr, capacity=200000)
            s = ctx.event_step(store, k)
            st.append({q: s[q] for q in keys})
        assert st[0]["status"] == 0 and st[0] == st[1]
