"""The cascade step as one persistent pass (children queued as they are written)
against the generation loop: the same particles, bit for bit, and the same
counts.  Sizes at the edges of a warp and of its event ring, a queue of one
chain and of many, each process alone, generations counted, and steps that
follow one another on one context (queue entries of earlier steps).  GPU only."""
import numpy as np
import pytest

from paper_2008_10468_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


def _sorted(a):
    o = np.argsort(a["id"], kind="stable")
    return {k: v[o] for k, v in a.items()}


@pytest.mark.parametrize("n,hot,cfg", [
    (1, 1.0, {}), (31, 1.0, {}), (33, 0.5, {"p_max": 0.9, "dt": 0.02}), (300, 0.5, {}),
    (300, 0.3, {"process_mask": 1}), (300, 0.3, {"process_mask": 2}), (5000, 0.2, {"recoil": False}),
    (70001, 0.02, {}), (70001, 0.0, {})])
def test_one_pass_equals_generations(n, hot, cfg):
    arr = I.clumped_mixed(n, 61, hot_fraction=hot)
    res = []
    for tail, passes in ((0, 64), (1 << 17, 64), (1 << 17, 63)):
        ctx = qed.Context(seed=29, max_passes=passes, **cfg)
        ctx.set_tail(tail)
        out = []
        for k in range(3):   # a large step, then one whose queue is smaller, then the first again
            a = arr if k != 1 else {f: v[: max(1, n // 3)] for f, v in arr.items()}
            store = qed.ParticleStore.from_numpy(a, capacity=n * 60 + 2000)
            st = ctx.event_step(store, 70 + k)
            assert st["status"] == 0 and st["count"] == store.n()
            out.append((st, _sorted(store.to_numpy())))
        res.append(out)
    cascade = cfg.get("process_mask", 3) == 3   # one process alone: no child has an event
    assert all(st["passes"] == 1 and st["tail"] == int(cascade) for st, _ in res[1])
    for other in res[1:]:
        for (sa, ga), (sb, gb) in zip(res[0], other):
            for k in ("substeps", "emissions", "pairs", "children", "plans", "candidates",
                      "max_N", "guard_hits", "count"):
                assert sa[k] == sb[k], (k, sa[k], sb[k])
            for k in ga:
                np.testing.assert_array_equal(ga[k], gb[k])
