"""The FP64 path stays bit-identical to the oracle where its integer quotients and roots take
their other branches (zeros, scales beyond 2^+-510, inadmissible states) and where con2prim
passes over inadmissible points unevaluated (bad warm starts, states next to v^2 = 1)."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import compare_bitwise
from paper_2212_00370_gb300 import rrmhd
from paper_2212_00370_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _states(n, seed):
    w = W.riemann_batch(n, seed=seed, nmin=2, nmax=2)
    return w, np.ascontiguousarray(w.V)


@pytest.mark.parametrize("case", ["zeros", "tiny", "huge", "mixed"])
def test_conversions_at_the_edges_of_the_integer_forms(case):
    torch = pytest.importorskip("torch")
    w, V = _states(500, 3)
    n = V.shape[1]
    rng = np.random.default_rng(4)
    if case == "zeros":      # fluid at rest, no field, no flux, in every combination
        for rows in (slice(1, 4), slice(5, 8), slice(9, 12)):
            V[rows] *= rng.integers(0, 2, (3, n))
    scale = {"zeros": 1.0, "tiny": 1e-160, "huge": 1e75, "mixed": 10.0 ** rng.uniform(-150, 70, n)}[case]
    V[0] *= scale
    V[4] *= scale
    V[8:] *= scale
    V[5:8] *= np.sqrt(scale)
    P = O.Params(gamma=w.gamma)
    ctx = rrmhd.Context([rrmhd.make_grid(1, (8,), (0.1,))], gamma=w.gamma)
    U = O.prim2con(V, P)
    compare_bitwise(ctx.prim2con(torch.tensor(V, device="cuda")).cpu().numpy(), U, "prim2con " + case)
    for guess in (None, O.prim_Z(V, P)):
        Vr, _, st = O.con2prim(U, P, guess)
        g = None if guess is None else torch.tensor(guess, device="cuda")
        Vg, sg = ctx.con2prim(torch.tensor(U, device="cuda"), g)
        compare_bitwise(sg.cpu().numpy(), st, "status " + case)
        ok = st == 0
        compare_bitwise(Vg.cpu().numpy()[:, ok], Vr[:, ok], "con2prim " + case)


@pytest.mark.parametrize("guess", [1e-12, 1e-3, 0.5, 2.0, 1e3, 1e12, -1.0, float("nan"), float("inf")])
def test_con2prim_from_bad_warm_starts(guess):
    torch = pytest.importorskip("torch")
    w, V = _states(2000, 5)
    n = V.shape[1]
    rng = np.random.default_rng(6)
    P = O.Params(gamma=w.gamma)
    U = O.prim2con(V, P)
    U[4] *= 1 - 10.0 ** rng.uniform(-12, 0, n)          # towards and past the admissible limit
    U[1:4] *= 1 + 10.0 ** rng.uniform(-12, -1, n)
    Z = guess * (U[0] + np.abs(U[4]))
    ctx = rrmhd.Context([rrmhd.make_grid(1, (8,), (0.1,))], gamma=w.gamma)
    Vg, sg = ctx.con2prim(torch.tensor(U, device="cuda"), torch.tensor(Z, device="cuda"))
    Vr, _, st = O.con2prim(U, P, Z)
    assert (st != 0).any() and ((st == 0).any() or guess == np.inf)  # inf: no root is found
    compare_bitwise(sg.cpu().numpy(), st, "status")
    ok = st == 0
    compare_bitwise(Vg.cpu().numpy()[:, ok], Vr[:, ok], "con2prim")
