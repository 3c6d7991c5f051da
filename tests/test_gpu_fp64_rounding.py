"""Rounding error of the FP64 stepper: over boxes of several spacings and
boundaries (mu = 1) its E is no further from the scheme in extended precision
than the scheme's plain restatement in float64, operation by operation, is."""
import math

import numpy as np
import pytest

from paper_2305_13419_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]


def _plain(w, state, steps, T):
    """E after `steps` steps in numpy type T."""
    n, N, per = w.n, w.storage_dims(), [b == "periodic" for b in w.bc]
    d, dt = [T(x) for x in w.d], T(w.courant / (W.C0 * math.sqrt(sum(1.0 / x ** 2 for x in w.d))))
    eps0, mu0, theta = T(W.EPS0), T(W.MU0), T(w.theta)
    at = [np.arange(N[a]).reshape([-1 if i == 2 - a else 1 for i in range(3)]) for a in range(3)]

    def mask(half):
        m = np.ones((N[2], N[1], N[0]), bool)
        for a in range(3):
            if not per[a]:
                m &= (at[a] < n[a]) & (half[a] | (at[a] >= 1))
        return m

    mE, mB = ([mask([(a == c) == e for a in range(3)]) for c in range(3)] for e in (True, False))

    def cells(x):   # a cell map on the storage points
        for a in range(3):
            if not per[a]:
                x = np.concatenate([x, np.take(x, [n[a] - 1], 2 - a)], 2 - a)
        return x.astype(T)

    def four(x, c):
        for b in ((c + 1) % 3, (c + 2) % 3):
            x = x + np.roll(x, 1, 2 - b)
        return x

    def edge(x, c):   # mean over the cells of the edge where it is not zero
        return four(x, c) / np.maximum(four((x > 0).astype(T), c), 1)

    lam = cells(w.lambda_L)
    kap = np.where(lam > 0, 1 / (np.where(lam > 0, lam, 1) ** 2 * mu0), T(0))
    ca, cb, kp = [], [], []
    for c in range(3):
        e = eps0 * four(cells(w.eps_r), c) / 4
        s = edge(cells(w.sigma), c) * dt / e
        ca.append((1 - (1 - theta) * s) / (1 + theta * s))
        cb.append(dt / e / (1 + theta * s))
        kp.append(np.where(mE[c], edge(kap, c), T(0)))
    prof, pb, pe = {}, {}, {}
    for a in range(3):
        if w.bc[a] == "cpml":
            cp = w.cpml[a]
            for half in (0, 1):
                x = at[a] + T(0.5) * half
                rho = np.maximum(np.maximum(cp.ncells - x, x - (n[a] - cp.ncells)) / T(cp.ncells), 0)
                s, al = T(cp.sigma_max) * rho ** T(cp.order), T(cp.alpha_max) * (1 - rho)
                b = np.exp(-(s + al) * dt / eps0)
                c_ = s * (b - 1) / np.where(s + al > 0, s + al, 1)
                prof[a, half] = np.where(rho > 0, b, 0), np.where(rho > 0, c_, 0)
            for c in range(3):
                if c != a:
                    pb[c, a] = pe[c, a] = np.zeros((N[2], N[1], N[0]), T)
    E, B, J = ([np.where(m, state[3 * k + c].astype(T), T(0)) for c, m in enumerate(ms)]
               for k, ms in enumerate((mE, mB, [k_ > 0 for k_ in kp])))
    sign = {(c, a): 1 if (a - c) % 3 == 1 else -1 for c in range(3) for a in range(3)}

    def dE(c, a):
        return (np.roll(E[3 - c - a], -1, 2 - a) - E[3 - c - a]) / d[a]

    def psi_b():
        for c, a in pb:
            b, c_ = prof[a, 1]
            pb[c, a] = np.where(mB[c], b * pb[c, a] + c_ * dE(c, a), T(0))

    def half_b():
        return [np.where(mB[c], B[c] - dt / 2 * sum(sign[c, a] * (dE(c, a) + pb.get((c, a), 0))
                                                    for a in range(3) if a != c), B[c]) for c in range(3)]

    psi_b()
    for _ in range(steps):
        B = half_b()
        J = [J[c] + dt / 2 * kp[c] * E[c] for c in range(3)]
        H = [b / mu0 for b in B]
        new = []
        for c in range(3):
            r = T(0)
            for a in range(3):
                if a != c:
                    v = (H[3 - c - a] - np.roll(H[3 - c - a], 1, 2 - a)) / d[a]
                    if (c, a) in pe:
                        b, c_ = prof[a, 0]
                        pe[c, a] = np.where(mE[c], b * pe[c, a] + c_ * v, T(0))
                        v = v + pe[c, a]
                    r = r + sign[c, a] * v
            new.append(np.where(mE[c], ca[c] * E[c] + cb[c] * (r - J[c]), E[c]))
        E = new
        J = [J[c] + dt / 2 * kp[c] * E[c] for c in range(3)]
        psi_b()
        B = half_b()
    return np.stack(E)


def test_error_is_no_larger_than_that_of_plain_float64():
    from paper_2305_13419_gb300 import twofluid as tf
    if np.finfo(np.longdouble).nmant <= 53:
        pytest.skip("needs a long double wider than double")
    rng = np.random.default_rng(6)
    mine, plain = [], []
    for i in range(8):
        bc = ("periodic",) * 3 if i % 2 else ("cpml", "pec", "cpml")
        w = W.random_box(n=(14, 12, 16), bc=bc, seed=i, d=tuple(rng.uniform(5e-9, 20e-9, 3)), theta=1.0,
                         lam_range=(60e-9, 90e-9), cpml_cells=5)
        st = W.random_state(i, w.storage_dims())
        keep = np.zeros(st[0].shape)
        keep[1:-2, 1:-2, 1:-2] = 1.0   # (the stepper takes a state as it is given: off the walls, no Js)
        st = [st[c] * (keep if c < 6 else 0.0) for c in range(9)]
        g = tf.Grid64.from_workload(w)
        for c in range(9):
            g.set_field(c, st[c])
        g.step(64)
        true = _plain(w, st, 64, np.longdouble)
        size = np.sqrt((true ** 2).sum())
        for out, E in ((mine, np.stack([g.field(c) for c in range(3)])), (plain, _plain(w, st, 64, np.float64))):
            out.append(float(np.sqrt(((E - true) ** 2).sum()) / size))
    assert max(mine) < 1e-13, mine   # the same scheme
    assert np.mean(mine) <= np.mean(plain), (mine, plain)
