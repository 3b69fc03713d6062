"""The windows in which the conversions take products on the integer pipes keep out what makes
a factor infinite or NaN: speeds of light and above, an infinite gamma (gamma/(gamma - 1) and
its inverse are then NaN).  Equal to the oracle bit for bit, NaN and infinities included."""
import numpy as np
import pytest

import oracle as O
from paper_2212_00370_gb300 import rrmhd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def fast_states(n, seed, field):
    """|v_k| < 1 and v^2 from just below 1 to 3, exactly 1 among them."""
    r = np.random.default_rng(seed)
    V = np.empty((12, n))
    V[0] = 10.0 ** r.uniform(-2, 1, n)
    V[4] = 10.0 ** r.uniform(-3, 1, n)
    V[5:8] = r.uniform(-1, 1, (3, n)) * field
    V[8] = 10.0 ** r.uniform(-3, 1, n)
    V[9:] = r.uniform(-0.5, 0.5, (3, n)) * V[8]
    d = r.normal(size=(3, n))
    d /= np.sqrt((d * d).sum(0))
    V[1:4] = d * (1 + r.choice([-1, 1], n) * 10.0 ** r.uniform(-17, -1, n))
    k = np.arange(n) % 4 == 0
    V[1:4, k] = r.choice([-1, 1], (3, k.sum())) * r.uniform(0.58, 1, (3, k.sum()))
    one = np.arange(n) % 16 == 1
    V[1:4, one] = np.array([0.6, 0.8, 0.0])[r.permutation(3)][:, None]
    V[1:4] = np.clip(V[1:4], -0.9999999, 0.9999999)
    return V


def same(a, b, what):
    assert np.array_equal(a, b, equal_nan=True), \
        f"{what}: {(~((a == b) | (np.isnan(a) & np.isnan(b)))).sum()} of {a.size} values differ"


@pytest.mark.parametrize("field", [0.0, 1.0])
def test_prim2con_at_the_speed_of_light(field):
    n, gamma = 20000, 4 / 3
    V = fast_states(n, 11, field)
    v2 = (V[1] * V[1] + V[2] * V[2]) + V[3] * V[3]
    assert (v2 == 1).sum() > 500 and (v2 > 1).sum() > 5000 and (v2 < 1).sum() > 5000
    U = O.prim2con(V, O.Params(gamma=gamma))
    assert np.isnan(U[0, v2 > 1]).all() and np.isinf(U[0, v2 == 1]).all()
    ctx = rrmhd.Context([rrmhd.make_grid(1, (n,), (1.0 / n,))], gamma=gamma)
    Vt = torch.tensor(V, device="cuda")
    same(ctx.prim2con(Vt).cpu().numpy(), U, "prim2con")
    ctx.set_state(Vt)
    same(ctx.get_state()[0].cpu().numpy(), U, "set_state")


@pytest.mark.parametrize("call", ["prim2con", "con2prim"])
def test_conversions_with_an_infinite_gamma(call):
    n, gamma = 100000, float("inf")
    r = np.random.default_rng(12)
    V = fast_states(n, 12, 1.0)
    V[1:4] *= r.uniform(0, 1, n)
    for k in (0, 4, 8):
        V[k] = 2.0 ** r.uniform(-20, 20, n)
    V[5:8] *= 2.0 ** r.uniform(-10, 10, n)
    P = O.Params(gamma=gamma)
    ctx = rrmhd.Context([rrmhd.make_grid(1, (8,), (0.1,))], gamma=gamma)
    if call == "prim2con":
        same(ctx.prim2con(torch.tensor(V, device="cuda")).cpu().numpy(), O.prim2con(V, P), call)
        return
    U = O.prim2con(V, O.Params(gamma=4 / 3))
    ok = np.isfinite(U).all(0)
    U = np.ascontiguousarray(U[:, ok])
    for guess in (None, U[0] * 2.0 ** r.uniform(-10, 10, ok.sum())):
        Vr, _, st = O.con2prim(U, P, guess)
        g = None if guess is None else torch.tensor(guess, device="cuda")
        Vg, sg = ctx.con2prim(torch.tensor(U, device="cuda"), g)
        assert (st != 0).all()          # the pressure is NaN: no state is recovered
        same(sg.cpu().numpy().astype(float), st.astype(float), "status")
        same(Vg.cpu().numpy(), np.zeros_like(Vr), "con2prim")
