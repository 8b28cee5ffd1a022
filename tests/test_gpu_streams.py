"""Steps of several contexts at once, each on its own stream and host thread.
Each persistent pass asks for all of the GPU, so some blocks of one may not be
resident while those of another wait: the resident ones must be able to end
their step without them.  Same rows and counts as alone.  GPU only."""
import threading

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


def _steps(arr, seed, nsteps, stream=None):
    out = []
    with torch.cuda.stream(stream or torch.cuda.current_stream()):
        ctx = qed.Context(seed=seed)
        for k in range(nsteps):
            store = qed.ParticleStore.from_numpy(arr, capacity=len(arr["px"]) * 20 + 20000)
            out.append((ctx.event_step(store, 90 + k), _sorted(store.to_numpy())))
        ctx.close()
    return out


@pytest.mark.parametrize("sizes", [(60000, 60000), (30000, 1000, 150000, 50)])
def test_concurrent_steps(sizes):
    nsteps = 12
    arrs = [I.clumped_mixed(n, 70 + k, hot_fraction=0.2) for k, n in enumerate(sizes)]
    alone = [_steps(a, 11 + k, nsteps) for k, a in enumerate(arrs)]
    torch.cuda.synchronize()
    got = [None] * len(sizes)

    def work(k, stream):
        got[k] = _steps(arrs[k], 11 + k, nsteps, stream)

    ts = [threading.Thread(target=work, args=(k, torch.cuda.Stream())) for k in range(len(sizes))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for a, g in zip(alone, got):
        assert g is not None
        for (sa, ra), (sg, rg) in zip(a, g):
            assert sa["status"] == 0 == sg["status"]
            for k in ("substeps", "emissions", "pairs", "children", "plans", "count"):
                assert sa[k] == sg[k], k
            for k in ra:
                np.testing.assert_array_equal(ra[k], rg[k], err_msg=k)
