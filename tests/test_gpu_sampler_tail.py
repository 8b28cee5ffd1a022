"""The tail pass of the sampler modes, in both of its forms (tails whose first
generation is below the line between them, and above), against the generations:
the same particles bit for bit, the same counts, and for the event-driven form
the same candidates (those up to an event).  The networks are trained until every
chi bin is usable, so that no e+- changes between sampler and rejection.  GPU
only."""
import numpy as np
import pytest

from paper_2008_10468_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402

TAIL_SMALL = 1 << 14   # rows of the tail's first generation at the line


def _sorted(a):
    o = np.argsort(a["id"], kind="stable")
    return {k: v[o] for k, v in a.items()}


@pytest.fixture(scope="module")
def weights():
    out = {}
    ctx = qed.Context(seed=1, sampler="event")
    for process in (qed.PROC_EMISSION, qed.PROC_PAIR):
        ctx.sampler_process(process)
        ctx.sampler_train(20081051, 1 << 26, batch=2048, lr=3e-3)
        out[process] = ctx.sampler_save()
    return out


@pytest.mark.parametrize("n,hot", [(3, 1.0), (4000, 0.05), (60000, 0.02), (60000, 0.12)])
@pytest.mark.parametrize("mode", [True, "event"])
def test_tail_forms_equal_generations(weights, mode, n, hot):
    arr = I.clumped_mixed(n, 83, hot_fraction=hot)
    res = []
    for tail in (0, 1 << 30):
        ctx = qed.Context(seed=37, sampler=mode, sampler_max_err=1e-3)
        for process, w in weights.items():
            if process == qed.PROC_EMISSION or mode == "event":
                ctx.sampler_process(process)
                ctx.sampler_load(w)
                ctx.sampler_evaluate()
        ctx.set_tail(tail)
        store = qed.ParticleStore.from_numpy(arr, capacity=n * 20 + 20000)
        st = ctx.event_step(store, 9)
        assert st["status"] == 0 and st["tail"] == int(tail > 0)
        res.append((st, _sorted(store.to_numpy())))
    (a, ga), (b, gb) = res
    if n == 60000:   # the children of the first generation, which the tail starts with
        one = qed.Context(seed=37, cascade=False)
        first = one.event_step(qed.ParticleStore.from_numpy(arr, capacity=n * 20), 9)["children"]
        assert (first < 0.8 * TAIL_SMALL) if hot == 0.02 else (first > 1.25 * TAIL_SMALL)
    keys = ["substeps", "emissions", "pairs", "children", "plans", "max_N", "count",
            "sampler_events", "sampler_pairs"] + (["candidates"] if mode == "event" else [])
    for k in keys:
        assert a[k] == b[k], (k, a[k], b[k])
    assert n < 100 or a["sampler_events"] > 0
    for k in ga:
        np.testing.assert_array_equal(ga[k], gb[k], err_msg=k)
