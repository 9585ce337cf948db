"""The level-ordered triangular solves over the forms their lanes-per-row rule
picks: narrow levels with short and long rows, and levels wide enough (more than
32 rows per SM) for four lanes per row in either precision, with 0 to 9
dependencies per row (empty, partial and several batches of every form)."""
import numpy as np
import pytest

from synth import BSRSystem, cartesian, random_bsr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2308_11892_gb300 as P
    return P


def two_levels(n, seed=31):
    """Rows 0..n/2-1 and n/2..n-1 coupled only across the halves, the second half's
    rows to 0..9 rows of the first and back: two levels of n/2 rows per triangle."""
    rng = np.random.default_rng(seed)
    h = n // 2
    A = np.zeros((h, 9), np.int64)
    for q in range(9):  # distinct columns per row
        A[:, q] = (np.arange(h) * 7 + q * 31 + 1) % h
    cnt = rng.integers(0, 10, h)
    keep = np.arange(9)[None, :] < cnt[:, None]
    r2, c1 = np.nonzero(keep)[0] + h, A[keep]
    rows = np.concatenate([np.arange(n), r2, c1])
    cols = np.concatenate([np.arange(n), c1, r2])
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order]
    vals = rng.uniform(-1, 1, (rows.size, 16))
    vals[rows == cols] += 40.0 * np.eye(4).ravel()
    rowptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(rows, minlength=n), out=rowptr[1:])
    return BSRSystem(n, rowptr.astype(np.int32), cols.astype(np.int32), vals,
                     rng.normal(size=4 * n), {})


SYSTEMS = {
    "one_cell": lambda: random_bsr(1),
    "narrow_short": lambda: cartesian(9, 7, 5, seed=3),
    "narrow_long": lambda: random_bsr(500, avg_offdiag=14.0, seed=4),
    "wide_mixed": lambda: two_levels(12000),
}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_level_solves_match_oracle(P, oracle_mod, monkeypatch, name, prec):
    import torch
    s = SYSTEMS[name]()
    o = oracle_mod.Oracle.from_system(s, precond=P.PREC_ILU).setup()
    r = np.random.default_rng(9).normal(size=4 * s.n_cells)
    outs = []
    for R in (0, 1):
        monkeypatch.setenv("CPTR_TRI_R", str(R))
        with P.Solver.from_system(s, precision=P.MIXED if prec == "mixed" else P.FP64,
                                  precond=P.PREC_ILU).setup() as g:
            if R == 0:
                assert P.cptr_get_info(g.h)["tri_schedule"] == 0
            out = torch.zeros(4 * s.n_cells, dtype=torch.float64, device="cuda")
            x = torch.from_numpy(r).cuda()
            torch.cuda.synchronize()
            P.cptr_apply(g.h, P.APPLY_ILU, x, out)
            torch.cuda.synchronize()
            outs.append(out.cpu().numpy())
    ref = o.ilu_apply(r)
    # FP64: the same sums up to contraction; mixed: FP32 factors and sums
    assert np.linalg.norm(outs[0] - ref) <= (1e-12 if prec == "fp64" else 1e-5) * np.linalg.norm(ref)
    np.testing.assert_array_equal(outs[0], outs[1])  # every schedule rounds alike
