"""The level-ordered triangular solves of lines and plane grids (rows of at most three
and five blocks), whose batches of dependencies are one and two long: the bits of the
cluster schedule, and the oracle's application to rounding."""
import numpy as np
import pytest

from synth import BSRSystem, cartesian

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2308_11892_gb300 as P
    return P


def both_ends():
    """Rows 0 and 1 couple to row 2 alone, and so on: two lower, then two upper blocks."""
    n = 300
    rows, cols = [], []
    for i in range(n):
        js = {i} | ({i - 2, i - 1} if i % 3 == 2 else {i - i % 3 + 2} & set(range(n)))
        rows += [i] * len(js)
        cols += sorted(js)
    rows, cols = np.array(rows), np.array(cols)
    v = np.random.default_rng(5).uniform(-1, 1, (rows.size, 16))
    v[rows == cols] += 6.0 * np.eye(4).ravel()
    rp = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=rp[1:])
    return BSRSystem(n, rp.astype(np.int32), cols.astype(np.int32), v,
                     np.random.default_rng(6).normal(size=4 * n), {})


SYSTEMS = {
    "two_cells": lambda: cartesian(1, 1, 2, seed=2),
    "line": lambda: cartesian(1, 1, 77, seed=3),
    "strip": lambda: cartesian(40, 2, 1, seed=4),
    "plane": lambda: cartesian(31, 23, 1, seed=5),
    "both_ends": both_ends,
}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_thin_levels(P, oracle_mod, monkeypatch, name, prec):
    import torch
    s = SYSTEMS[name]()
    o = oracle_mod.Oracle.from_system(s, precond=P.PREC_ILU).setup()
    r = np.random.default_rng(9).normal(size=4 * s.n_cells)
    outs = []
    for R in (0, 1):
        monkeypatch.setenv("CPTR_TRI_R", str(R))
        with P.Solver.from_system(s, precision=P.MIXED if prec == "mixed" else P.FP64,
                                  precond=P.PREC_ILU).setup() as g:
            out = torch.zeros(4 * s.n_cells, dtype=torch.float64, device="cuda")
            x = torch.from_numpy(r).cuda()
            torch.cuda.synchronize()
            P.cptr_apply(g.h, P.APPLY_ILU, x, out)
            torch.cuda.synchronize()
            outs.append(out.cpu().numpy())
    ref = o.ilu_apply(r)
    # FP64: the same sums up to contraction; mixed: FP32 factors and sums
    assert np.linalg.norm(outs[0] - ref) <= (1e-12 if prec == "fp64" else 1e-5) * np.linalg.norm(ref)
    np.testing.assert_array_equal(outs[0], outs[1])
