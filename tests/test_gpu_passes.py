"""Steps in place (a B pass and an E pass per step, what tf_step does on grids
of up to some 80 million points) and many steps per launch (grids with a
narrow cross section) give the same bits as the staged single-step
kernel: fields, probe DFTs and series, on every boundary kind, on rows that
end inside a thread's four points, with sources and probes at the walls,
varying mu, both edge rules and split calls, and in any mix with staged steps
on one handle."""
import numpy as np
import pytest

from paper_2305_13419_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

P, C, W_, M = "periodic", "cpml", "pec", "mur"
# size, boundaries, edge rule, theta, range of mu
CASES = [
    ((1, 1, 300), (P, P, M), 0, 1.0, (1.0, 1.0)),
    ((1, 1, 2), (P, P, M), 0, 1.0, (1.0, 1.0)),
    ((2, 3, 5), (P, P, P), 1, 0.5, (1.0, 2.0)),
    ((4, 4, 130), (P, P, M), 0, 1.0, (1.0, 1.0)),
    ((5, 7, 3), (W_, W_, M), 0, 0.5, (1.0, 2.0)),
    ((33, 17, 9), (W_, P, W_), 1, 1.0, (1.0, 1.0)),
    ((66, 34, 33), (C, C, C), 0, 1.0, (1.0, 1.0)),
    ((67, 33, 30), (C, P, C), 0, 0.5, (1.0, 2.0)),
    ((70, 29, 31), (P, C, M), 1, 1.0, (1.0, 1.0)),
    ((131, 21, 18), (W_, C, P), 0, 1.0, (1.0, 1.0)),
    ((96, 50, 40), (P, P, P), 0, 0.5, (1.0, 1.0)),
    ((65, 8, 64), (P, W_, C), 0, 1.0, (1.0, 2.0)),
    # narrow cross sections (many steps per launch), at the ends of their range
    ((1, 1, 4), (P, P, P), 0, 1.0, (1.0, 1.0)),
    ((1, 1, 700), (P, P, C), 0, 1.0, (1.0, 1.0)),
    ((3, 5, 90), (P, P, C), 0, 0.5, (1.0, 1.0)),
    ((127, 1, 40), (P, P, W_), 0, 1.0, (1.0, 1.0)),
    ((4, 32, 33), (P, P, M), 1, 1.0, (1.0, 1.0)),
    ((9, 9, 61), (P, W_, M), 0, 1.0, (1.0, 1.0)),
    ((14, 7, 50), (W_, W_, P), 0, 0.5, (1.0, 1.0)),
    ((2, 2, 300), (W_, P, M), 0, 1.0, (1.0, 1.0)),
]


def _workload(n, bc, rule, theta, mu):
    w = W.random_box(n=n, bc=bc, seed=sum(n), theta=theta, mu_range=mu, cpml_cells=max(1, min(4, min(n) // 2)))
    w.edge_rule = rule
    f = W.C0 / (20 * w.d[2])
    hi = w.storage_dims()
    w.sources = [W.Source(comp=c, lo=(n[0] // 3, 0, n[2] // 2), hi=(n[0] // 3 + 5, n[1], n[2] // 2 + 2), amp=0.3 + c,
                          kind=c, f=f, t0=3e-16, tw=1e-16) for c in range(3)]
    pts = [(0, 0, 0), (hi[0] - 1, hi[1] - 1, hi[2] - 1), (n[0] // 2, n[1] // 2, n[2] // 2)]
    w.probes = [W.Probe(comp=c, p=p, freqs=np.linspace(0.5 * f, 2 * f, 3 + 7 * c), n0=5 * c, series=50)
                for c, p in enumerate(pts)]
    return w


def _grid(w, staged):
    from paper_2305_13419_gb300 import twofluid as tf
    g = tf.Grid.from_workload(w)
    g.set_two_step(False)
    if staged:
        g.set_wait_limit(1 << 21)   # a limit of the handle's own: the staged kernel
    st = W.random_state(11, w.storage_dims())
    for c in range(9):
        g.set_field(c, st[c].astype(np.float32))
    return g


def _same(a, b, w, n):
    for c in range(9):
        assert np.array_equal(a.field(c), b.field(c)), c
    for p in range(len(w.probes)):
        assert np.array_equal(a.probe_dft(p), b.probe_dft(p)), p
        assert np.array_equal(a.probe_series(p, n), b.probe_series(p, n)), p


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[0])) + "-" + "-".join(c[1]))
def test_passes_give_the_bits_of_staged_steps(case):
    w = _workload(*case)
    ref = _grid(w, True)
    ref.step(41)
    ref.sync()
    for chunks in ([41], [1, 2, 38]):
        g = _grid(w, False)
        for n in chunks:
            g.step(n)
        g.sync()
        _same(g, ref, w, 41)


def test_passes_with_mu_in_blocks():
    """mu constant over most tile-planes but not over the grid."""
    w = _workload((96, 48, 20), (P, P, C), 0, 1.0, (1.0, 2.0))
    w.eps_r[:], w.sigma[:], w.lambda_L[:] = 2.5, 2e5, 40e-9
    w.mu_r[:] = 1.7
    w.mu_r[:, :, :2] = 1.3
    ref = _grid(w, True)
    ref.step(15)
    g = _grid(w, False)
    g.step(15)
    _same(g, ref, w, 15)


@pytest.mark.parametrize("case", [CASES[6], CASES[8], CASES[14], CASES[17]], ids=["cpml", "mur", "narrow-cpml", "narrow-mur"])
def test_passes_and_staged_steps_mix(case):
    """In place, staged and two-step passes in turn on one handle."""
    w = _workload(*case)
    ref = _grid(w, True)
    ref.step(26)
    g = _grid(w, False)
    g.step(5)
    g.set_wait_limit(1 << 21)
    g.step(3)
    g.set_wait_limit(None)
    g.step(4)
    g.set_two_step(8)   # (the narrow grids have no box: they stay as they are)
    g.step(5)
    g.set_two_step(False)
    g.step(9)
    g.sync()
    _same(g, ref, w, 26)


@pytest.mark.parametrize("sizes,count", [((24, 33, 40), 5), ((96, 104), 2)])
def test_batches_in_place_and_staged(sizes, count):
    """tf_batch_run grid by grid in place against its one launch per step over
    all grids, sources and probes and a narrow grid among them."""
    from paper_2305_13419_gb300 import twofluid as tf
    ws = [_workload((n, sizes[0] + i, sizes[-1] - i), (C, P, C), 0, 1.0, (1.0, 1.0))
          for i, n in enumerate((sizes * count)[:count])]
    ws.append(_workload((2, 3, 40), (P, P, M), 0, 1.0, (1.0, 1.0)))
    runs = []
    for staged in (False, True):
        grids = [_grid(w, staged) for w in ws]
        tf.batch_run(grids, 35)
        tf.batch_run(grids, 6)
        runs.append(grids)
    for w, a, b in zip(ws, *runs):
        assert a.level == 41
        _same(a, b, w, 41)


@pytest.mark.parametrize("cap,max_probes,mu", [(71, 1, (1.0, 1.0)), (71, 3, (1.0, 2.0)), (72, 2, (1.0, 2.0))])
def test_adjoint_checkpoints_leave_the_forward_state(cap, max_probes, mu):
    """The adjoint's checkpoints hold every part, a series of odd length among
    them, and a restore leaves all buffers as a run without it does."""
    from paper_2305_13419_gb300 import twofluid as tf
    w = _workload((40, 9, 11), (C, P, C), 0, 1.0, mu)
    w.probes = w.probes[:1]
    runs = []
    for adjoint in (True, False):
        g = tf.Grid.from_workload(w, series_capacity=cap, max_probes=max_probes)
        if adjoint:
            g.adjoint(50, 0, 0, segment=9)
        else:
            g.step(50)
        g.step(12)   # the state is also good to go on from, in place and staged
        g.set_wait_limit(1 << 21)
        g.step(7)
        g.sync()
        runs.append(g)
    _same(runs[0], runs[1], w, 50)


def test_probe_without_frequencies_reads_an_empty_spectrum():
    w = _workload((20, 9, 11), (P, P, C), 0, 1.0, (1.0, 1.0))
    w.probes = [W.Probe(comp=0, p=(3, 4, 5), freqs=np.zeros(0), series=9), w.probes[1]]
    g = _grid(w, False)
    g.step(9)
    assert g.probe_dft(0).size == 0 and g.probe_series(0, 9).size == 9
    assert g.probe_dft(1).size > 0


@pytest.mark.parametrize("case", [((205, 131, 140), (C, P, C), 0, 1.0, (1.0, 1.0)),
                                  ((203, 130, 141), (W_, C, M), 1, 0.5, (1.0, 1.0)),
                                  ((300, 201, 90), (P, W_, W_), 0, 1.0, (1.0, 2.0)),
                                  ((64, 41, 1500), (P, C, M), 0, 1.0, (1.0, 1.0))],
                         ids=["cpml", "mur", "pec-mu", "long"])
def test_windows_of_planes_give_the_bits_of_staged_steps(case):
    """Grids large enough to be stepped window by window, several steps each:
    probes on the first, the last and a middle plane, group ends inside a
    window's depth."""
    w = _workload(*case)
    ref = _grid(w, True)
    ref.step(41)
    g = _grid(w, False)
    for n in (1, 2, 33, 5):
        g.step(n)
    g.sync()
    _same(g, ref, w, 41)


def test_windows_of_planes_keep_the_history_of_the_adjoint():
    """E at every level, written window by window, against staged steps' copies."""
    from paper_2305_13419_gb300 import twofluid as tf
    n = (205, 131, 140)
    w = _workload(n, (C, P, C), 0, 1.0, (1.0, 1.0))
    w.probes = [W.Probe(comp=0, p=(n[0] // 3 + 7, n[1] // 2, n[2] // 2 + 1), freqs=w.probes[0].freqs)]
    out = []
    for staged in (True, False):
        g = tf.Grid.from_workload(w)
        g.set_two_step(False)
        if staged:
            g.set_wait_limit(1 << 21)
        out.append(g.adjoint(40, 0, 0, segment=9))
    (J, eps, lam), (J1, eps1, lam1) = out
    assert J > 0 and J == J1
    assert torch.equal(eps, eps1) and torch.equal(lam, lam1)
