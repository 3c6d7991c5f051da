"""Mur walls of grids that take many steps per launch: lengths at which a wall
is the first plane past a window (a multiple of the planes that a CTA owns),
and windows that own one plane, in full launches and in the short last one.
The same bits as the staged single-step kernel."""
import pytest

from test_gpu_passes import M, P, W_, _grid, _same, _workload

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("n,chunks", [((8, 8, 1000), (40, 3)), ((8, 8, 2048), (40,)), ((9, 9, 1000), (40, 1)),
                                      ((4, 4, 600), (2, 2, 1)), ((4, 4, 128), (40, 7)), ((1, 1, 254), (1, 1)),
                                      ((1, 1, 508), (1, 2, 3)), ((1, 1, 1000), (3, 3)), ((16, 8, 60), (40, 2, 1)),
                                      ((9, 9, 100), (40, 4)), ((5, 5, 100), (45, 1, 4)), ((2, 7, 2), (9, 1)),
                                      ((1, 1, 4480), (40,))],
                         ids=lambda v: "x".join(map(str, v)))
@pytest.mark.parametrize("bcy", [P, W_])
def test_walls_next_to_the_last_owned_plane(n, chunks, bcy):
    if bcy == W_ and n[1] == 1:
        pytest.skip("a column has no inner points between walls")
    w = _workload(n, (P, bcy, M), 0, 1.0, (1.0, 1.0))
    steps = sum(chunks)
    for p in w.probes:
        p.series = steps
    ref, g = _grid(w, True), _grid(w, False)
    ref.step(steps)
    for m in chunks:
        g.step(m)
    g.sync()
    _same(g, ref, w, steps)
