"""Read-back converts the stored Bt and Jt to SI by a product that is rounded
once, as FP64 arithmetic would: ties that a product of two FP32 parts gets
wrong, and magnitudes down to the subnormal numbers, where its parts run out
of bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu,
              pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")]

C0, EPS0 = 299792458.0, 8.8541878128e-12
# a time step and a Js whose conversion lies that close to a tie
TIES = [("0x1.dd42d3dd89a14p-51", "0x1.fa8ca6p+13"), ("0x1.2eafdc58d777dp-60", "0x1.8469ccp+23"),
        ("0x1.cf996ecc92017p-59", "0x1.c2e9bp+21"), ("0x1.1580b8e6b6bd5p-51", "0x1.c518f4p+14")]


@pytest.mark.parametrize("nx", [7, 70])
@pytest.mark.parametrize("dt,js", TIES, ids=[t[0] for t in TIES])
def test_conversion_to_si_is_rounded_once(dt, js, nx):
    from paper_2305_13419_gb300 import twofluid as tf
    dt, js = float.fromhex(dt), float.fromhex(js)
    d = 4.0 * C0 * dt
    g = tf.Grid((nx, 60, 50), (d, d, d), dt=dt)
    one = np.ones((50, 60, nx), np.float32)
    g.set_materials(one, one, 20.0 * d * one, 0.0 * one)
    rng = np.random.default_rng(3)
    for comp in (3, 4, 5, 6, 7, 8):
        to = C0 if comp < 6 else dt / EPS0
        v = rng.standard_normal(g.shape) * 10.0 ** rng.uniform(-46, -28, g.shape)
        v[:, ::2] = rng.standard_normal(v[:, ::2].shape) * (1e-9 if comp < 6 else js)
        v[:, 1, :] = js * 2.0 ** rng.integers(-8, 8, v[:, 1, :].shape)
        v[0, 0, :5] = 0.0, -0.0, np.inf, -np.inf, np.nan
        v = v.astype(np.float32)
        g.set_field(comp, v)
        with np.errstate(invalid="ignore", over="ignore"):
            held = (v.astype(np.float64) * to).astype(np.float32)
            want = (held.astype(np.float64) * (1.0 / C0 if comp < 6 else EPS0 / dt)).astype(np.float32)
        assert np.array_equal(g.field(comp), want, equal_nan=True), comp


@pytest.mark.parametrize("bc", [("periodic", "periodic", "periodic"), ("pec", "periodic", "mur"), ("periodic", "pec", "pec")],
                         ids="-".join)
@pytest.mark.parametrize("nx", [7, 33, 140])
def test_integer_level_b_rounds_every_product_and_sum(nx, bc):
    """B^n = B^{n-1/2} - curl E / 2 of the stored arrays, formed in FP32 one
    operation at a time, whichever kernel reads the row."""
    from paper_2305_13419_gb300 import twofluid as tf
    from paper_2305_13419_gb300 import workloads as W
    w = W.random_box(n=(nx, 9, 11), bc=bc, seed=nx)
    st = W.random_state(4, w.storage_dims())
    g = tf.Grid.from_workload(w)
    for c in range(9):
        g.set_field(c, st[c].astype(np.float32))
    g.step(2)
    blob = g.save_checkpoint()
    pitch = int(blob[20:24].view(np.int32)[0])   # after the magic and the three sizes
    raw = blob[256:].view(np.float32)[:6 * pitch * g.N[1] * g.N[2]].reshape(6, g.N[2], g.N[1], pitch)[..., :g.N[0]]
    E, B = raw[:3], raw[3:]
    r = [np.float32(C0 * g.dt / w.d[a]) for a in range(3)]
    for c in range(3):
        acc = np.zeros(g.shape, np.float32)
        held = np.zeros(g.shape, bool)
        for a in range(3):
            if bc[a] != "periodic":   # off the axis: the half positions; along it: off both walls
                at = np.arange(g.N[a]).reshape([-1 if i == 2 - a else 1 for i in range(3)])
                held |= (at == w.n[a]) | ((at == 0) if a == c else False)
            if a == c:
                continue
            t = r[a] * (np.roll(E[3 - c - a], -1, 2 - a) - E[3 - c - a])
            acc = acc + (t if (a - c) % 3 == 1 else -t)
        b = np.where(held, B[c], B[c] - np.float32(0.5) * acc)
        want = (b.astype(np.float64) * (1.0 / C0)).astype(np.float32)
        assert np.array_equal(g.field(3 + c), want), c
