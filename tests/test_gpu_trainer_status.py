"""A wait that runs out in one of the trainer's tensor-core layers: calls that synchronise fail, calls that
do not write NaN, no Adam step is taken, and the next calls are as good as before.  The waits' limit is set
to no poll at all; the products are still waited for, so the GPU stays usable."""
import ctypes as C

import numpy as np
import pytest

import helm6_inputs as inputs
from oracle import cnn

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def wait_limit(lib, tr, polls):
    f = getattr(lib, "_ZN5helm614cnn_wait_limitEP17helm6_cnn_traineri")  # helm6::cnn_wait_limit
    f.argtypes, f.restype = [C.c_void_p, C.c_int], None
    f(tr._tr, polls)


@pytest.mark.parametrize("shape", [(1, 5, 8, 12), (2, 4, 6, 40)])  # runs and bricks
def test_a_wait_that_runs_out(shape):
    from paper_1212_1397_gb300 import build, helm6
    build.build()
    lib = helm6.load()
    th = cnn.init_params(inputs.standard_normal(41, cnn.n_params())).astype(np.float32)
    x = torch.from_numpy(inputs.standard_normal(42, int(np.prod(shape)) * 2).reshape(shape + (2,)).astype(np.float32)).cuda()
    with helm6.Trainer(*shape, th) as tr:
        y = tr.forward(x)
        loss, g = tr.gradient(x, x)
        assert torch.isfinite(y).all() and torch.isfinite(g).all()
        wait_limit(lib, tr, 0)
        assert torch.isnan(tr.forward(x)).all()
        bad = torch.zeros(helm6.CNN_NPARAMS, device="cuda")
        ptr = lambda t: C.c_void_p(t.data_ptr())
        assert lib.helm6_cnn_gradient(tr._tr, ptr(x), ptr(x), ptr(bad), None) == 0  # no loss, no synchronisation
        assert torch.isnan(bad).all()
        with pytest.raises(helm6.Helm6Error):
            tr.gradient(x, x)
        with pytest.raises(helm6.Helm6Error):
            tr.step(x, x, 0.1)
        assert tr.step(x, x, 0.1, want_loss=False) is None
        wait_limit(lib, tr, 1 << 22)
        with pytest.raises(helm6.Helm6Error):  # the step that was not taken
            tr.params()
        assert np.array_equal(tr.params(), th)
        assert torch.equal(tr.forward(x), y)
        loss2, g2 = tr.gradient(x, x)
        assert loss2 == loss and torch.equal(g2, g)
        tr.step(x, x, 0.1)
        assert not np.array_equal(tr.params(), th)
