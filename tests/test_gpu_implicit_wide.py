"""Warps of the implicit solve with every mix of cells: hard ones (10^2 and more evaluations),
easy ones, cells without opacity, lanes without a cell, instances that are not advanced, and in
the fallback passes cells that are not updated again.  When four cells or fewer are left in a
warp its idle lanes evaluate for them; blocks of 8 threads never do that, so the two must agree
bit for bit, in both precisions; the FP64 form also equals the oracle."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import compare_bitwise, gpu_context
from paper_2212_00370_gb300 import rrmhd
from paper_2212_00370_gb300 import workloads as W
from test_gpu_fallback import HARD

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HDT = 0.3


@pytest.fixture(scope="module")
def cells():
    """2000 states; their opacities (none in every 7th); evaluations of R and status of each solve."""
    w = W.riemann_batch(1000, seed=9, nmin=2, nmax=2)
    P = O.Params(gamma=w.gamma)
    V = np.ascontiguousarray(w.V)
    kappa, sigma = w.kappa.copy(), w.sigma.copy()
    kappa[::7] = sigma[::7] = 0.0
    U, Z = O.prim2con(V, P), O.prim_Z(V, P)
    ev, st = np.zeros(V.shape[1], int), np.zeros(V.shape[1], int)
    for i in range(V.shape[1]):
        s = O.Stats()
        st[i] = O.implicit(U[:, i:i + 1], kappa[i:i + 1], sigma[i:i + 1], HDT, P, Z[i:i + 1], stats=s)[2][0]
        ev[i] = s.imp_resid
    return V, U, Z, kappa, sigma, ev, st, P


def mixed(cells, n):
    """n cells, the hardest that are solved and some of the others in turn."""
    kappa, ev, st = cells[3], cells[5], cells[6]
    hard = [i for i in np.argsort(-ev, kind="stable") if st[i] == 0]
    failed, none = np.flatnonzero(st != 0), np.flatnonzero(kappa == 0)
    easy = np.flatnonzero((ev > 0) & (ev < 10))
    ix = []
    for j in range(n):
        k = j // 4
        ix.append([hard[k], easy[k], none[k], failed[k % len(failed)] if k % 2 else hard[200 + k]][j % 4])
    assert ev[hard[0]] > 200 and (n < 3 or (kappa[ix] == 0).any()) and (n < 8 or (st[ix] != 0).any())
    return np.array(ix)


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 33, 100])
def test_mixed_cells_equal_the_oracle(cells, n):
    V, U, Z, kappa, sigma, _, _, P = cells
    ix = mixed(cells, n)
    Us = np.ascontiguousarray(U[:, ix])
    Ur, Vr, st = O.implicit(Us, kappa[ix], sigma[ix], HDT, P, Z[ix])
    ctx = rrmhd.Context([rrmhd.make_grid(1, (n,), (0.01,))], gamma=P.gamma)
    dev = [torch.tensor(a, device="cuda") for a in (Us, Z[ix], kappa[ix], sigma[ix])]
    ctx.set_opacity(dev[2], dev[3])
    Ug, Vg, sg = (x.cpu().numpy() for x in ctx.implicit_source(HDT, dev[0], dev[1]))
    ok = st == 0
    assert ok.any()
    compare_bitwise(sg, st, "status")
    compare_bitwise(Ug[:, ok], Ur[:, ok], "U")
    compare_bitwise(Vg[:, ok], Vr[:, ok], "V")


@pytest.mark.parametrize("precision", ["fp64", "fp32_bulk"])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 33, 100])
def test_wide_rounds_equal_blocks_without_them(cells, n, precision):
    """One-cell instances (their fluxes cancel): a step is the solve of each cell."""
    V, _, _, kappa, sigma, _, _, P = cells
    ix = mixed(cells, n)
    grid = {"ndim": 1, "n": (1, 1, 1), "dx": (1.0, 1.0, 1.0), "bc": ("outflow",) * 3}
    w = W.Workload("cells", [grid] * n, np.ascontiguousarray(V[:, ix]), kappa[ix], sigma[ix],
                   np.full(n, np.inf), P.gamma)
    ref = None
    for shape in (dict(cell_block=8), dict(cell_block=128), dict(cell_block=32, cell_persistent=1)):
        ctx = gpu_context(w, precision=precision)
        ctx.set_tuning(lanes=1, cell_per_thread=1, **{"cell_persistent": 0, **shape})
        ctx.imex_step(3)
        got = [x.cpu().numpy() for x in ctx.get_state()] + [ctx.inst_status(), ctx.get_times()[0]]
        ctx.close()
        if ref is None:
            ref = got
            assert (ref[2] == 0).any()
            continue
        for a, b, what in zip(got, ref, ("U", "V", "status", "t")):
            compare_bitwise(a, b, f"{what} under {shape}")


@pytest.mark.parametrize("precision", ["fp64", "fp32_bulk"])
def test_fallback_of_mixed_instances_equals_each_alone(precision):
    """Instances that need fallback passes next to short ones, one that has reached its end, one
    that starts with an inadmissible cell; the last block of cells is not full."""
    hard = W.riemann_batch().subset(HARD[:2] + HARD[6:8])
    short = W.riemann_batch(6, seed=31, nmin=3, nmax=21)
    order = [(short, 0), (hard, 0), (short, 1), (short, 2), (hard, 2), (short, 3), (hard, 1), (short, 4),
             (hard, 3), (short, 5)]
    one = [src.subset([i]) for src, i in order]
    one[3].V[8, 1] = 0.0
    one[5].t_end[0] = 0.0
    w = W.Workload("mixed", [o.grids[0] for o in one], np.ascontiguousarray(np.concatenate([o.V for o in one], 1)),
                   np.concatenate([o.kappa for o in one]), np.concatenate([o.sigma for o in one]),
                   np.concatenate([o.t_end for o in one]), hard.gamma)
    assert w.ncells % 32 != 0

    def run(x):
        ctx = gpu_context(x, precision=precision, lanes=1)
        ctx.imex_step(13)
        got = [a.cpu().numpy() for a in ctx.get_state()] + [ctx.inst_status(), ctx.get_times()[0]]
        ctx.close()
        return got

    U, V, st, t = run(w)
    off = w.cell_offsets()
    for j, o in enumerate(one):
        Uj, Vj, sj, tj = run(o)
        s = slice(off[j], off[j + 1])
        assert st[j] == sj[0] and t[j] == tj[0]
        compare_bitwise(U[:, s], Uj, f"instance {j} U")
        compare_bitwise(V[:, s], Vj, f"instance {j} V")
    assert t[5] == 0.0 and (st[[1, 4, 6, 8]] == 0).any()
