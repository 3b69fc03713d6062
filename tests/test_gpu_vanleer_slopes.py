"""VanLeer slopes where the product of the two differences is not a normal number: the faces
keep the limiter's own order of operations there, 2 dL dR/(dL + dR), and the oracle's bits."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import compare_bitwise, gpu_context, oracle_grid, oracle_params
from paper_2212_00370_gb300 import workloads as W

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solver", ["pvm", "radhll"])
@pytest.mark.parametrize("lo, hi", [(-165, -145), (-322, -300), (-322, -1)])
def test_slopes_next_to_the_smallest_numbers(lo, hi, solver):
    n = 400
    r = np.random.default_rng(-lo - hi)
    V = np.zeros((12, n))
    V[0] = r.uniform(0.5, 2, n)
    V[4] = r.uniform(0.5, 2, n)
    V[8] = r.uniform(1, 2, n)
    for k in (1, 2, 3, 5, 6, 7, 9, 10, 11):  # monotone, over the decades lo..hi
        V[k] = r.choice([-1, 1]) * np.sort(10.0 ** r.uniform(lo, hi, n))[:: r.choice([-1, 1])]
    d = np.diff(V, axis=1)
    p = np.abs(d[:, :-1] * d[:, 1:])
    if hi == -145:
        assert ((p > 0) & (p < 2.0 ** -1022)).sum() > 500
    w = W.Workload("slopes", [W.grid1d(n)], V, np.ones(n), np.ones(n), np.array([1.0]), 4 / 3)
    P = oracle_params(w, solver=solver)
    F = O.face_flux(oracle_grid(w.grids[0]), 0, O.prim2con(V, P), V, w.kappa, w.sigma, P)
    ctx = gpu_context(w, solver=solver)
    compare_bitwise(ctx.flux_sweep(0).cpu().numpy(), F.reshape(12, -1), "faces")
