"""The two-kernel training step and the three kernels of large batches form the same
sums in the same order: the same weights bit for bit after one step, where Adam
sees the signs of the gradient, and after several, where it sees their sizes.
Ragged tiles, one chunk of 32 tiles and several, both networks.  GPU only."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2008_10468_gb300 import qed  # noqa: E402


def _train(batch, steps, three, process):
    ctx = qed.Context(seed=3, sampler="event")
    f = qed.lib().qed_test_train_three
    f.argtypes, f.restype = [C.c_void_p, C.c_int], C.c_int
    assert f(ctx._h, int(three)) == qed.QED_OK
    ctx.sampler_process(process)
    loss = ctx.sampler_train(77, steps * batch, batch=batch, lr=3e-3)
    return loss, ctx.sampler_save()


@pytest.mark.parametrize("batch", [64, 65, 127, 1000, 2047, 2048, 2049, 2112, 4160, 8192, 19455,
                                   19456])
@pytest.mark.parametrize("process", [qed.PROC_EMISSION, qed.PROC_PAIR])
def test_both_forms_give_the_same_weights(batch, process):
    for steps in (1, 2, 7):
        l2, two = _train(batch, steps, False, process)
        l3, three = _train(batch, steps, True, process)
        np.testing.assert_array_equal(two.view(np.uint32), three.view(np.uint32),
                                      err_msg="%d steps" % steps)
        # the loss is summed by atomic adds of at most 1216 partial sums, in any
        # order: 1216 2^-24 = 7e-5 of it
        assert abs(l2 - l3) <= 1e-4 * l3
