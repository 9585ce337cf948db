"""What is singular is decided on the roundings of the definition: products and sums
rounded one by one, no fused multiply-add.  Matrices whose elimination cancels
exactly, or only just does not, are refused exactly when the definition refuses
them."""
import numpy as np
import pytest

from synth import cartesian, knn, random_bsr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    import paper_2308_11892_gb300 as P
    return P


def _setup_status(P, n, rp, ci, v, **kw):
    g = P.Solver(n, np.asarray(rp, np.int32), np.asarray(ci, np.int32), v, **kw)
    try:
        g.setup()
        return P._lib.OK
    except P.CPTRError as e:
        return e.status
    finally:
        g.close()


@pytest.mark.parametrize("kind", ["repeated", "scaled", "equal_blocks"])
def test_ilu_pivot_block_that_cancels(P, oracle_mod, kind):
    """Two cells whose block rows are multiples of each other: the second pivot block
    is A_11 - (k A_00 inv(A_00)) A_01, zero up to rounding."""
    refused = 0
    for seed in range(100):
        r = np.random.default_rng(seed)
        B = r.uniform(-1, 1, (4, 4)) + 2 * np.eye(4)
        C = B.copy() if kind == "equal_blocks" else r.uniform(-1, 1, (4, 4))
        k = 3.0 if kind == "scaled" else 1.0
        v = np.stack([b.reshape(16) for b in (B, C, k * B, k * C)])
        rp, ci = [0, 2, 4], [0, 1, 0, 1]
        try:
            oracle_mod.Oracle(np.array(rp, np.int32), np.array(ci, np.int32), v,
                              precond=oracle_mod.PREC_ILU).setup()
            want = P._lib.OK
        except RuntimeError:
            want = P._lib.ERR_BREAKDOWN
            refused += 1
        assert _setup_status(P, 2, rp, ci, v, precond=P.PREC_ILU) == want, seed
    assert 0 < refused < 100  # both answers occur


def dense_blocks(sizes, seed):
    """Cells in groups with dense patterns of the given sizes, not coupled to others."""
    r = np.random.default_rng(seed)
    rp, ci, v, i0 = [0], [], [], 0
    for s in sizes:
        for i in range(s):
            ci += list(range(i0, i0 + s))
            b = r.uniform(-1, 1, (s, 4, 4))
            b[i] += (3.0 + s) * np.eye(4)
            v.append(b.reshape(s, 16))
            rp.append(len(ci))
        i0 += s
    return i0, rp, ci, np.concatenate(v)


# dense groups: from ten cells on a row's shared columns do not fit its list, beside
# shorter rows in the same warp; 33 cells and more: the kernel of one row per warp
@pytest.mark.parametrize("name", ["grid", "cloud", "random", "dense_16", "dense_32", "dense_33"])
def test_ilu_factors_have_the_definition_s_bits(P, oracle_mod, name):
    if name.startswith("dense"):
        n, rp, ci, v = dense_blocks([1, 2, 9, 10, 11, 5, int(name[6:]), 3, 12], seed=8)
        rp, ci = np.asarray(rp, np.int32), np.asarray(ci, np.int32)
    else:
        s = {"grid": lambda: cartesian(11, 9, 7, pe=5.0, seed=3), "cloud": lambda: knn(9, 8, 7, seed=4),
             "random": lambda: random_bsr(300, avg_offdiag=14.0, seed=5)}[name]()
        n, rp, ci, v = s.n_cells, s.rowptr, s.col, s.vals
    o = oracle_mod.Oracle(rp, ci, v, precond=oracle_mod.PREC_ILU).setup()
    with P.Solver(n, rp, ci, v, precond=P.PREC_ILU).setup() as g:
        F = g.copy(0, P.COPY_ILU, np.float64, 16 * len(ci))
    np.testing.assert_array_equal(F.ravel(), np.asarray(o.ilu_factors()).ravel())
