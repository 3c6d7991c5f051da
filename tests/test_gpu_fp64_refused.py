"""A refused tf64_set_materials call leaves the FP64 stepper's materials as
they were."""
import numpy as np
import pytest

from paper_2305_13419_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("mu", [(1.0, 2.0), (1.0, 1.0)], ids=["mu", "uniform"])
def test_a_refused_call_keeps_the_materials(mu):
    from paper_2305_13419_gb300 import twofluid as tf
    w = W.random_box(n=(9, 7, 11), bc=("periodic", "pec", "cpml"), seed=3, mu_range=mu, cpml_cells=3)
    st = W.random_state(13, w.storage_dims())
    bad = np.array(w.eps_r)
    bad.flat[0 if mu[1] > 1 else -1] = -1.0
    other = np.ones_like(w.mu_r) if mu[1] > 1 else np.full_like(w.mu_r, 1.5)
    out = []
    for refused in (False, True):
        g = tf.Grid64.from_workload(w)
        if refused:
            with pytest.raises(tf.TFError) as ex:
                g.set_materials(bad, other, w.lambda_L, w.sigma)
            assert ex.value.status == tf.TF_EINVAL
        for c in range(9):
            g.set_field(c, st[c])
        g.step(20)
        g.sync()
        out.append([g.field(c) for c in range(9)])
    for c in range(9):
        assert np.array_equal(out[0][c], out[1][c]), c
