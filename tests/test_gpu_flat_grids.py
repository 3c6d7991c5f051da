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
