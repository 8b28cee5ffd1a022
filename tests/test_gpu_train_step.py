"""The two-kernel training step against the three-kernel one it replaces for
small batches, through the entry point, at ragged and whole tiles and chunks and
at the size where the kernels change.  GPU only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


@pytest.mark.parametrize("batch", [64, 65, 1000, 2047, 2048, 2049, 4160, 19456])
def test_training_is_reproducible_and_learns(batch):
    # every tile count the two-kernel step takes, ragged last tiles, one and
    # several chunks of 32 tiles: the same call gives the same bits, and a
    # short training lowers the loss
    def train(samples):
        ctx = qed.Context(seed=3, sampler="event")
        loss = ctx.sampler_train(77, samples, batch=batch, lr=3e-3)
        return loss, ctx.sampler_save()

    l1, a = train(batch)
    l2, b = train(24 * batch)
    l3, c = train(24 * batch)
    assert np.isfinite(b).all() and abs(l2 - l3) <= 1e-5 * l2
    np.testing.assert_array_equal(b, c)
    assert l2 < l1


def test_first_step_agrees_with_the_large_batch_kernels():
    # 304 tiles are the largest two-kernel step of a 152-SM GPU, one sample more
    # takes the large-batch kernels.  Adam's first step is lr times the sign of
    # the gradient (up to eps).  The two batches share all samples but one, of
    # weight 1 / 19457, against a batch gradient of about 1 / sqrt(19457) of a
    # sample's: a sign differs for about 0.8 sqrt(19457) / 19457 = 0.6% of the
    # weights; five times that is allowed.
    def step(b):
        ctx = qed.Context(seed=3, sampler="event")
        r = np.random.default_rng(1)
        th = (r.uniform(-1, 1, qed.SAMPLER_PARAMS) / 8.0).astype(np.float32)
        ctx.sampler_load(th)
        ctx.sampler_train(5, b, batch=b, lr=1e-3)
        return ctx.sampler_save() - th

    tiles = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    d, ref = step(64 * tiles), step(64 * tiles + 1)
    assert (np.abs(d) <= 1.01e-3).all()
    assert (np.sign(d) != np.sign(ref)).mean() < 0.03
