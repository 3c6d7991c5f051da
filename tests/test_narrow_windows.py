"""Windows of planes that step by themselves (the narrow kernel): which planes
are still right after a launch, by tracking what every value was formed from.
A plane of E or B is right if all it reads is; what lies past a window's end
is not.  Every plane must be stored once, by a window in which it is right."""
import numpy as np
import pytest


def _right_after(steps, z0, z1, nz, mur):
    """Planes of [z0, z1) whose E and B are right after `steps` steps, walls at 0 and nz."""
    k = np.arange(z0, z1)
    e, b = np.ones(k.size, bool), np.ones(k.size, bool)
    inner = (k > 0) & (k < nz)
    for _ in range(steps):
        up = np.append(e[1:], False)
        b = np.where(k < nz, b & e & up, b)   # B_k from E_k, E_k+1
        old, dn = e, np.insert(b[:-1], 0, False)
        e = np.where(inner, e & b & dn, e)    # E_k from B_k, B_k-1
        e = np.where(k == 0, e & b, e)        # (its z component)
        if mur:                               # E of a wall from E of the plane next to it, old and new
            for w, i in ((0, 1), (nz, nz - 1)):
                if z0 <= w < z1:
                    at, ok = w - z0, z0 <= i < z1
                    e[at] = e[at] and ok and old[i - z0] and e[i - z0]
    return e & b


@pytest.mark.parametrize("mur", [False, True], ids=["held", "mur"])
@pytest.mark.parametrize("window", [8, 9, 10, 11, 16, 23, 32])
def test_every_plane_is_stored_once_and_right(window, mur):
    for steps in range(1, (window - 1) // 2 + 1):
        own = window - 2 * steps
        for nz in (*range(2, 3 * own + 6), 8 * own, 8 * own + 1):
            stored = np.zeros(nz + 1, int)
            for first in range(0, nz if mur else nz + 1, own):
                z0, z1 = max(first - steps, 0), min(first - steps + window, nz + 1)
                right = _right_after(steps, z0, z1, nz, mur)
                for k in range(z0, z1):
                    owner = min(max(k, 1), nz - 1) if mur else k   # a Mur wall goes with the plane next to it
                    if first <= owner < first + own:
                        stored[k] += 1
                        assert right[k - z0], (steps, nz, k)
            assert (stored == 1).all(), (steps, nz)
