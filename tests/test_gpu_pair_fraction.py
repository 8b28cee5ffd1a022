"""Pair events whose electron fraction is exactly 0, which a network with large
weights can return (its sigmoid underflows): a pair like any other, one electron
and one positron with the photon's momentum between them.  GPU only."""
import numpy as np
import pytest

from paper_2008_10468_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


@pytest.mark.parametrize("cascade", [False, True])
@pytest.mark.parametrize("bias", [-400.0, 400.0])   # fractions 0 and 1
def test_fraction_at_an_end(cascade, bias):
    arr = I.clumped_mixed(3000, 19, hot_fraction=1.0)
    photons = arr["type"] == qed.PHOTON
    arr = {k: v[photons] for k, v in arr.items()}
    n = len(arr["px"])
    ctx = qed.Context(seed=8, sampler="event", sampler_max_err=2.0, cascade=cascade, dt=0.05)
    for process, b4 in ((qed.PROC_EMISSION, 0.0), (qed.PROC_PAIR, bias)):
        w = np.zeros(qed.SAMPLER_PARAMS, np.float32)
        w[-1] = b4
        ctx.sampler_process(process)
        ctx.sampler_load(w)
        ctx.sampler_evaluate()
    store = qed.ParticleStore.from_numpy(arr, capacity=n * 300)
    st = ctx.event_step(store, 2)
    assert st["status"] == 0 and st["sampler_pairs"] > 20
    got = store.to_numpy()
    assert st["count"] == n + st["children"] == len(got["id"])
    assert st["children"] == st["emissions"] + 2 * st["pairs"]
    assert len(np.unique(got["id"])) == len(got["id"])
    kinds = {t: int((got["type"] == t).sum()) for t in (qed.ELECTRON, qed.POSITRON)}
    assert kinds[qed.ELECTRON] == kinds[qed.POSITRON] == st["pairs"]
    if not cascade:
        assert st["emissions"] == 0
        # of a sampled pair the one lepton has nothing of the photon's momentum,
        # the other all of it (short plans decay by rejection)
        for t, none in ((qed.ELECTRON, bias < 0), (qed.POSITRON, bias > 0)):
            rows = got["type"] == t
            p = np.stack([got[k][rows] for k in ("px", "py", "pz")])
            assert (np.abs(p).max(axis=0) == 0).sum() == (st["sampler_pairs"] if none else 0)
        gone = got["type"][:n] == qed.REMOVED
        assert gone.sum() == st["pairs"]
        np.testing.assert_allclose(np.abs(got["px"][n:]).sum(dtype=np.float64),
                                   np.abs(arr["px"][gone]).sum(dtype=np.float64), rtol=1e-6)
