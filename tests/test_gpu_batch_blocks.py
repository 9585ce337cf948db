"""Batched solves on clusters of 1, 2, 4 and 8 blocks: the number of blocks only
deals the rows, so every size gives the same bits, for systems smaller than one
block's share, with a handful of rows per level and with several slices."""
import numpy as np
import pytest

from synth import cartesian, knn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2308_11892_gb300 as P
    return P


def _solve(P, systems, **kw):
    solvers = [P.Solver.from_system(s, **kw).setup() for s in systems]
    try:
        xs = [np.zeros(4 * s.n_cells) for s in systems]
        _, infos = P.cptr_solve_batch([g.h for g in solvers], [s.rhs for s in systems], xs)
        return xs, [i["iters"] for i in infos]
    finally:
        for g in solvers:
            g.close()


@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(precision=1, e1=-1),
                                dict(precond=2, restart=7), dict(nu_pre=2, nu_post=0)],
                         ids=["fp64", "mixed", "cpr", "ilu_restart", "sweeps"])
def test_cluster_size_does_not_change_the_result(P, monkeypatch, kw):
    systems = [cartesian(3, 2, 2, seed=61), knn(16, 14, 9, pe=5.0, seed=62),
               cartesian(20, 13, 9, pe=30.0, seed=63)]
    monkeypatch.setenv("CPTR_BATCH_BLOCKS", "1")
    ref, its = _solve(P, systems, **kw)
    for s, x in zip(systems, ref):
        r = s.rhs - _mv(s, x)
        assert np.linalg.norm(r) <= 1.001e-6 * np.linalg.norm(s.rhs)
    for blocks in ("2", "4", "8", None):  # None: by the rule, from the systems' sizes
        if blocks:
            monkeypatch.setenv("CPTR_BATCH_BLOCKS", blocks)
        else:
            monkeypatch.delenv("CPTR_BATCH_BLOCKS")
        xs, it2 = _solve(P, systems, **kw)
        assert it2 == its
        for a, b in zip(xs, ref):
            np.testing.assert_array_equal(a, b)


def _mv(s, x):
    rows = np.repeat(np.arange(s.n_cells), np.diff(s.rowptr))
    y = np.zeros((s.n_cells, 4))
    np.add.at(y, rows, np.einsum("bij,bj->bi", s.vals.reshape(-1, 4, 4), x.reshape(-1, 4)[s.col]))
    return y.ravel()


def test_wait_limit_is_reported(P, monkeypatch):
    """A dependency wait that runs out ends the batched solve with an error status,
    and the contexts solve again with the default limit."""
    monkeypatch.setenv("CPTR_BATCH_BLOCKS", "4")
    s = knn(16, 14, 9, pe=5.0, seed=62)
    with P.Solver.from_system(s, precision=1).setup() as g:
        x = np.zeros(4 * s.n_cells)
        P.cptr_set_spin_limit(g.h, 1)
        with pytest.raises(P.CPTRError) as e:
            P.cptr_solve_batch([g.h], [s.rhs], [x])
        assert e.value.status == P.ERR_TIMEOUT
        P.cptr_set_spin_limit(g.h, 0)
        x[:] = 0.0
        st, _ = P.cptr_solve_batch([g.h], [s.rhs], [x])
        assert st == 0
        assert np.linalg.norm(s.rhs - _mv(s, x)) <= 1.001e-6 * np.linalg.norm(s.rhs)
