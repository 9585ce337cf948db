"""The setup's row kernels, each forced on whole hierarchies: every choice adds a
row's terms in the definition's order, so all of them give the default's
hierarchy bit for bit, and the default's is the oracle's."""
import numpy as np
import pytest

from synth import cartesian, knn

pytestmark = pytest.mark.gpu

SYSTEMS = {
    "knn": lambda: knn(11, 9, 7, seed=21),
    "advective": lambda: cartesian(18, 14, 9, pe=100.0, seed=22),
}


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2308_11892_gb300 as P
    return P


def hierarchy(P, s, **kw):
    out = []
    with P.Solver.from_system(s, **kw).setup() as g:
        lev = g.levels()
        for l, i in enumerate(lev):
            out += [g.copy(l, P.COPY_A_ROWPTR, np.int32, i["n"] + 1),
                    g.copy(l, P.COPY_A_COL, np.int32, i["nnz"]),
                    g.copy(l, P.COPY_A_VAL, np.float64, i["nnz"])]
            if l < len(lev) - 1:
                out += [g.copy(l, P.COPY_CF, np.int32, i["n"]),
                        g.copy(l, P.COPY_P_ROWPTR, np.int32, i["n"] + 1),
                        g.copy(l, P.COPY_P_COL, np.int32, i["nnzP"]),
                        g.copy(l, P.COPY_P_VAL, np.float64, i["nnzP"])]
    return out


# path 4: every row starts in the smallest table (most move up class by class),
# 5: in the tables of 512 columns, 6: in the block-wide ones, 1: the ordered-table
# block kernel; pmax 1 and 12: rows of P of one entry and longer than a lane group
@pytest.mark.parametrize("pmax", [1, 4, 12])
@pytest.mark.parametrize("path", ["1", "4", "5", "6"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_spgemm_classes(P, monkeypatch, name, path, pmax):
    s = SYSTEMS[name]()
    ref = hierarchy(P, s, pmax=pmax)
    monkeypatch.setenv("CPTR_SPGEMM_PATH", path)
    got = hierarchy(P, s, pmax=pmax)
    assert len(got) == len(ref)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)


# path 3, 4, 5: every F point starts in the first, second and third class of the
# lane-group kernels (rows that do not fit move up), 1: wide blocks
@pytest.mark.parametrize("pmax", [1, 4, 12])
@pytest.mark.parametrize("path", ["1", "3", "4", "5"])
@pytest.mark.parametrize("name", list(SYSTEMS))
def test_interp_classes(P, monkeypatch, name, path, pmax):
    s = SYSTEMS[name]()
    ref = hierarchy(P, s, pmax=pmax)
    monkeypatch.setenv("CPTR_INTERP_PATH", path)
    got = hierarchy(P, s, pmax=pmax)
    assert len(got) == len(ref)
    for a, b in zip(got, ref):
        np.testing.assert_array_equal(a, b)
