"""The one-launch conjugate gradients (systems up to 311,296 rows) at the sizes
where its layout changes: single rows, odd tails, the edges of its 64-, 128-
and 192-, 256- and 512-row blocks and of its warps, and the first size past it.

A misaligned x takes the per-iteration kernels for every size; they form the
same sums in another order, so on these well-conditioned systems (diagonal
dominance puts the eigenvalues in [0.1, 2.05 * 18 + 0.1], a condition number
below 400) both stop at the same test of convergence, 8 iterations apart at
most, with residuals at rtol and solutions within 400 * 2 rtol of each other."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RTOL = 1e-12


@pytest.fixture(scope="module")
def ph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    return ph


def cu(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def banded_spd(n, offsets, seed):
    """Symmetric, strictly diagonally dominant by a factor 1.05, columns sorted."""
    rng = np.random.default_rng(seed)
    A = sp.csr_matrix((n, n))
    for o in offsets:
        if o < n:
            A = A + sp.diags(rng.uniform(-1.0, 1.0, n - o), o, shape=(n, n))
    A = sp.csr_matrix(A + A.T)
    A = sp.csr_matrix(A + sp.diags(1.05 * np.asarray(abs(A).sum(axis=1)).ravel() + 0.1))
    A.sort_indices()
    return A


@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 64, 65, 9727, 9728, 9729, 19456, 19457, 38911, 38912, 38913, 200003, 311295,
                               311296, 311297])
@pytest.mark.parametrize("offsets", [(1, 7, 50), (1, 2, 3, 5, 9, 17, 33, 65, 129, 257)])
def test_loop_solve_matches_per_iteration_kernels(ph, n, offsets):
    if len(offsets) > 3 and n not in (65, 9729, 38913):
        pytest.skip("rows wider than the ELL copy: one size of each layout")
    A = banded_spd(n, offsets, n)
    b = np.random.default_rng(n + 1).standard_normal(n)
    rp, ci, va, bd = cu(A.indptr.astype(np.int32)), cu(A.indices.astype(np.int32)), cu(A.data), cu(b)
    x0, it0, rr0, _ = ph.ph_solve_pcg(rp, ci, va, bd, rtol=RTOL, maxit=5000)
    buf = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    x1, it1, rr1, _ = ph.ph_solve_pcg(rp, ci, va, bd, rtol=RTOL, maxit=5000, x=buf[1:])
    assert abs(it0 - it1) <= 8 and rr0 <= RTOL and rr1 <= RTOL
    x0, x1 = x0.cpu().numpy(), x1.cpu().numpy()
    assert np.linalg.norm(A @ x0 - b) <= 10 * RTOL * np.linalg.norm(b)
    assert np.linalg.norm(x0 - x1) <= 800 * RTOL * np.linalg.norm(x1)
    if n <= ph.PH_PCG_NOALLOC_MAX_N:  # the CSR arrays and the four-vector workspace: the same bits
        x2, it2, rr2, _ = ph.ph_solve_pcg_noalloc(rp, ci, va, bd, rtol=RTOL, maxit=5000)
        assert it2 == it0 and rr2 == rr0 and np.array_equal(x2.cpu().numpy(), x0)


def test_loop_solve_iteration_cap_and_resume(ph):
    """Caps that are not multiples of 8, and more iterations than one launch
    makes (4096), against the same solve with a larger cap."""
    n = 3001
    A = sp.csr_matrix(sp.diags([-np.ones(n - 1), np.full(n, 2.0), -np.ones(n - 1)], [-1, 0, 1]))
    b = np.random.default_rng(5).standard_normal(n)
    rp, ci, va, bd = cu(A.indptr.astype(np.int32)), cu(A.indices.astype(np.int32)), cu(A.data), cu(b)
    for cap in (1, 7, 13, 4096, 4100):
        _, it, rr, code = ph.ph_solve_pcg(rp, ci, va, bd, rtol=0.0, maxit=cap, check=False)
        assert it == cap and code == 7 and np.isfinite(rr)
    x, it, rr, code = ph.ph_solve_pcg(rp, ci, va, bd, rtol=1e-10, maxit=20000)
    assert code == 0 and np.linalg.norm(A @ x.cpu().numpy() - b) <= 1e-8 * np.linalg.norm(b)
