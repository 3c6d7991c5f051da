"""Grids whose planes are large: passes in windows of the fewest planes they
take (fewer than the steps a window is moved down by), whole passes where a
window would be smaller.  The same bits as the staged single-step kernel."""
import pytest

from test_gpu_passes import C, M, P, W_, _grid, _same, _workload

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("case", [((701, 690, 12), (C, P, M), 0, 1.0, (1.0, 1.0)),
                                  ((500, 401, 21), (W_, C, C), 1, 0.5, (1.0, 2.0)),
                                  ((1001, 700, 9), (P, C, C), 0, 1.0, (1.0, 1.0)),
                                  ((1300, 1300, 2), (P, W_, M), 0, 0.5, (1.0, 1.0))],
                         ids=["windows-of-4", "windows-of-11", "whole", "whole-2"])
def test_flat_grids_give_the_bits_of_staged_steps(case):
    w = _workload(*case)
    ref = _grid(w, True)
    ref.step(41)
    g = _grid(w, False)
    for n in (1, 2, 33, 5):
        g.step(n)
    g.sync()
    _same(g, ref, w, 41)


def _uniform(n, bc, varying, default):
    from paper_2305_13419_gb300 import twofluid as tf
    from paper_2305_13419_gb300 import workloads as W
    d = (10e-9, 12e-9, 8e-9)
    cpml = tuple(W.default_cpml(6, d[a], 1e12) if bc[a] == C else None for a in range(3))
    gen = torch.Generator(device="cuda").manual_seed(5)
    g = tf.Grid(n, d, 1.0, bc, cpml, courant=0.9)
    cells = (n[2], n[1], n[0])
    eps = torch.full(cells, 2.5, device="cuda")
    if varying:
        eps += torch.rand(cells, generator=gen, device="cuda")
    g.set_materials(eps, torch.ones_like(eps), torch.zeros_like(eps), torch.zeros_like(eps))
    if not default:
        g.set_two_step(False)
    for c in range(6):
        g.set_field(c, (torch.rand(g.shape, generator=gen, device="cuda") - 0.5) * W.FIELD_SCALE[c])
    return g


def _same_on_device(g, h):
    a, b = (torch.empty(x.shape, device="cuda") for x in (g, h))
    for c in range(6):
        g.field(c, out=a)
        h.field(c, out=b)
        assert torch.equal(a, b), c


@pytest.mark.parametrize("n,bc,varying,two", [((512, 512, 128), (C, C, P), False, True), ((512, 512, 128), (C, C, P), True, False),
                                              ((256, 512, 128), (C, C, P), False, False), ((512, 512, 128), (P, C, P), False, False),
                                              ((800, 800, 80), (W_, W_, W_), False, True), ((512, 512, 128), (C, C, C), False, False),
                                              ((1000, 1000, 30), (C, C, C), False, False)])
def test_where_two_step_passes_pay(n, bc, varying, two):
    """tf_step's choice between steps in place and two-step passes where
    neither was asked for, and the same bits either way."""
    grids = [_uniform(n, bc, varying, default) for default in (True, False)]
    for g in grids:
        g.step(5)
        g.sync()
    assert [g.two_step_box()[1] for g in grids] == [two, False]
    _same_on_device(*grids)


@pytest.mark.parametrize("n,bc", [((700, 700, 80), (C, C, C)), ((512, 512, 128), (C, C, P))])
def test_short_calls_mix_the_routes(n, bc):
    """Calls of one step (whole passes), of two (a two-step pass) and of more
    in turn, against one call in place."""
    g, ref = _uniform(n, bc, False, True), _uniform(n, bc, False, False)
    for m in (1, 2, 3, 1, 4, 2):
        g.step(m)
    ref.step(13)
    g.sync()
    ref.sync()
    _same_on_device(g, ref)


def test_a_captured_call_runs_in_place():
    """A call that would take two-step passes, captured on a handle that has
    stepped in place only (no work lists yet)."""
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        g = _uniform((512, 512, 128), (C, C, P), False, True)
        g.step(1)
        g.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        g.step(2)
    graph.replay()
    torch.cuda.synchronize()
    ref = _uniform((512, 512, 128), (C, C, P), False, False)
    ref.step(3)
    ref.sync()
    assert g.level == 3
    _same_on_device(g, ref)
