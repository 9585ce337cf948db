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


def gauss_jordan(A):
    """The definition of the coarsest inverse: [A | I], partial pivoting (largest |a|,
    the first on ties), every product and difference rounded; None when singular."""
    n = len(A)
    a = np.concatenate([A, np.eye(n)], axis=1)
    for k in range(n):
        p = k + int(np.argmax(np.abs(a[k:, k])))
        if not abs(a[p, k]) > 0.0:
            return None
        a[[k, p]] = a[[p, k]]
        a[k] = a[k] / a[k, k]
        f = a[:, k].copy()
        f[k] = 0.0
        a = a - f[:, None] * a[k][None, :]
    return a[:, n:]


def pressure_system(L):
    """4x4 blocks with L in the first unknown and the identity in the others, so that
    the first stage's scalar operator is L itself."""
    n = len(L)
    i, j = np.nonzero((L != 0) | np.eye(n, dtype=bool))
    v = np.zeros((i.size, 4, 4))
    v[:, 0, 0] = L[i, j]
    v[i == j] += np.diag([0.0, 1.0, 1.0, 1.0])
    rp = np.zeros(n + 1, np.int32)
    np.cumsum(np.bincount(i, minlength=n), out=rp[1:])
    return n, rp, j.astype(np.int32), v.reshape(-1, 16)


def neumann(nx, ny, seed):
    """Five-point operator without a boundary condition: its rows sum to zero."""
    r = np.random.default_rng(seed)
    n = nx * ny
    L = np.zeros((n, n))
    for i in range(n):
        for j in ([i + 1] if (i + 1) % nx else []) + ([i + nx] if i + nx < n else []):
            L[i, j] = L[j, i] = -r.uniform(0.5, 2.0)
    for i in range(n):
        for j in np.nonzero(L[i])[0]:
            if j != i:
                L[i, i] -= L[i, j]
    return L


def test_coarsest_operator_that_cancels(P):
    answers = set()
    for seed in range(200):
        r = np.random.default_rng(seed)
        L = neumann(int(r.integers(2, 8)), int(r.integers(2, 8)), seed)
        want = P._lib.OK if gauss_jordan(L) is not None else P._lib.ERR_BREAKDOWN
        answers.add(want)
        assert _setup_status(P, *pressure_system(L), precond=P.PREC_FIRST, e1=-1) == want, seed
    assert len(answers) == 2


# one, two and 17 CTAs' worth of columns, slices with and without a remainder, the
# largest matrix of the cluster (609) and the one-block kernel's smallest
@pytest.mark.parametrize("n", [1, 15, 16, 17, 100, 209, 609, 610])
def test_coarsest_inverse_has_the_definition_s_bits(P, n):
    import torch
    r = np.random.default_rng(n)
    A = r.uniform(-1, 1, (n, n))
    A[r.uniform(size=(n, n)) < 0.5] = 0.0
    A[np.arange(n), np.arange(n)] = r.uniform(-1, 1, n)  # rows are exchanged
    want = gauss_jordan(A)
    cols = sorted({0, n // 3, n // 2, n - 1})
    with P.Solver(*pressure_system(A), precond=P.PREC_FIRST, e1=-1, max_coarse=1024).setup() as g:
        assert len(g.levels()) == 1
        for c in cols:
            b = torch.zeros(n, dtype=torch.float64, device="cuda")
            b[c] = 1.0
            x = torch.zeros_like(b)
            torch.cuda.synchronize()
            P.cptr_apply(g.h, P.APPLY_VCYCLE, b, x)
            torch.cuda.synchronize()
            np.testing.assert_array_equal(x.cpu().numpy(), want[:, c])
