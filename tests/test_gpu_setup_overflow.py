"""Rows that no class of the setup's row kernels holds: they go to the kernels with
tables in global memory, whose rows the others' equal bit for bit."""
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


def hierarchy(P, s, **kw):
    out = []
    with P.Solver.from_system(s, precond=P.PREC_FIRST, **kw).setup() as g:
        lev = g.levels()
        for l, i in enumerate(lev):
            out.append([g.copy(l, P.COPY_A_ROWPTR, np.int32, i["n"] + 1),
                        g.copy(l, P.COPY_A_COL, np.int32, i["nnz"]),
                        g.copy(l, P.COPY_A_VAL, np.float64, i["nnz"])])
            if l < len(lev) - 1:
                out[-1] += [g.copy(l, P.COPY_P_ROWPTR, np.int32, i["n"] + 1),
                            g.copy(l, P.COPY_P_COL, np.int32, i["nnzP"]),
                            g.copy(l, P.COPY_P_VAL, np.float64, i["nnzP"])]
    return out


def same(a, b):
    assert len(a) == len(b)
    for x, y in zip(a, b):
        for u, v in zip(x, y):
            np.testing.assert_array_equal(u, v)


def line_with_dense_row(n, strength, seed=1):
    """A line of cells, the last one coupled to all others."""
    s = cartesian(1, 1, n, seed=seed)
    r = np.random.default_rng(seed)
    cut = s.rowptr[n - 1]
    add = np.arange(n - 2)
    v = -strength * r.uniform(0.5, 1.0, (n - 2, 1)) * np.eye(4).ravel()
    last = s.vals.reshape(-1, 16)[cut:].copy()
    last[-1] += strength * n * np.eye(4).ravel()
    rp = s.rowptr.copy()
    rp[n] = cut + n
    assert rp[n] - rp[n - 1] == n
    return BSRSystem(n, rp, np.concatenate([s.col[:cut], add, s.col[cut:]]).astype(np.int32),
                     np.concatenate([s.vals.reshape(-1, 16)[:cut], v, last]), s.rhs, {})


def test_product_row_wider_than_every_table(P, monkeypatch):
    s = line_with_dense_row(40000, 1e-4)  # (weak couplings: a short row of P)
    got = hierarchy(P, s, e1=-1)
    rp, ci, _, prp, pci, _ = got[0]
    cols = np.unique(np.concatenate([pci[prp[j]:prp[j + 1]] for j in ci[rp[-2]:]]))
    assert cols.size > 8192  # 32 warps with 256 slots each cannot hold the row
    monkeypatch.setenv("CPTR_SPGEMM_PATH", "3")
    same(got, hierarchy(P, s, e1=-1))


# more than 128 strong F neighbours, more than 1536 terms: dense random patterns
@pytest.mark.parametrize("deg", [40.0, 90.0, 200.0])
def test_interpolation_row_larger_than_every_class(P, monkeypatch, deg):
    s = random_bsr(500, avg_offdiag=deg, seed=int(deg))
    got = hierarchy(P, s)
    monkeypatch.setenv("CPTR_INTERP_PATH", "2")
    same(got, hierarchy(P, s))
