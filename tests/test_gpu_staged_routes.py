"""The staged kernels on grids that would step in place (a wait limit of the
handle's own keeps them staged) against steps in place: the batch's one launch
per step over several replays of its captured graph and the launches that
remain, with grids at different levels and buffer parities, and the
single-step kernel's work-item lengths."""
import numpy as np
import pytest

from test_gpu_batch import _variants
from test_gpu_two_step import CASES
from paper_2305_13419_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _staged(w):
    from paper_2305_13419_gb300 import twofluid as tf
    g = tf.Grid.from_workload(w)
    g.set_two_step(False)
    g.set_wait_limit(1 << 21)
    return g


def _same(a, b, w):
    for c in range(9):
        assert np.array_equal(a.field(c), b.field(c)), (w.name, c)
    for p in range(len(w.probes)):
        assert np.array_equal(a.probe_dft(p), b.probe_dft(p)), (w.name, p)


@pytest.mark.parametrize("first", [3, 4])
def test_staged_batch_replays_and_remainder(first):
    from paper_2305_13419_gb300 import twofluid as tf
    ws = _variants()
    batch = [_staged(w) for w in ws]
    batch[0].step(first)
    tf.batch_run(batch[1:], first)
    tf.batch_run(batch[2:], 1)          # the first two stay a level behind
    tf.batch_run(batch, 150 - first)    # two replays of 64 steps, the rest launched one by one
    for i, (w, g) in enumerate(zip(ws, batch)):
        g.sync()
        n = 150 + (i >= 2)
        assert g.level == n
        ref = tf.Grid.from_workload(w)
        ref.step(n)
        _same(g, ref, w)


@pytest.mark.parametrize("planes", [8, 12, 16])
@pytest.mark.parametrize("name", ["cpw-small", "cpml-xz-periodic-y", "periodic-xy-mur-z"])
def test_staged_item_lengths_give_the_bits_of_steps_in_place(name, planes):
    from paper_2305_13419_gb300 import twofluid as tf
    w = CASES[name]()
    st = W.random_state(7, w.storage_dims())
    ref, g = tf.Grid.from_workload(w), _staged(w)
    g.set_item_planes(planes)
    for x in (ref, g):
        if not name.startswith("cpw"):
            for c in range(9):
                x.set_field(c, st[c].astype(np.float32))
        x.step(23)
        x.sync()
    _same(g, ref, w)
