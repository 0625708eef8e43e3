"""A block of the one-launch conjugate gradients that never arrives: every other
block's bounded wait runs out, the solve reports PH_ERR_TIMEOUT, gives back its
memory and leaves the context as it was.  One block and many, both layouts of
the rows, both preconditioners, the refined and the allocation-free solve."""
import numpy as np
import pytest

import meshgen
from tests.test_gpu_solve_loop import banded_spd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def cu(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.fixture(scope="module")
def ph():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    yield ph
    ph.ph_test_pcg_loop(0)


def check(ph, solve):
    """solve() -> (x, status name): a time-out with the hook, and without it the
    bits of a solve that was never interrupted."""
    x0, s0 = solve()
    torch.cuda.synchronize()
    before = ph.ph_pool_in_use()
    x0 = x0.clone()
    ph.ph_test_pcg_loop(2)
    try:
        _, s1 = solve()
    finally:
        ph.ph_test_pcg_loop(0)
    torch.cuda.synchronize()
    assert s0 == "PH_OK" and s1 == "PH_ERR_TIMEOUT"
    assert ph.ph_pool_in_use() == before
    x2, s2 = solve()
    assert s2 == "PH_OK" and torch.equal(x2, x0)


@pytest.mark.parametrize("n", [33, 9729, 40001])
def test_jacobi(ph, n):
    A = banded_spd(n, (1, 7, 50), n)
    rp, ci, va = cu(A.indptr.astype(np.int32)), cu(A.indices.astype(np.int32)), cu(A.data)
    b = cu(np.random.default_rng(n).standard_normal(n))
    for f in (ph.ph_solve_pcg, ph.ph_solve_pcg_noalloc):
        def solve():
            x, _, _, code = f(rp, ci, va, b, rtol=1e-10, maxit=2000, check=False)
            return x, ph.ph_status_string(code)
        check(ph, solve)


@pytest.mark.parametrize("m", [2, 15])
def test_schwarz_and_refined(ph, m):
    coord, tet = meshgen.kuhn_cube(m)
    mesh = ph.Mesh(cu(coord), cu(tet.astype(np.int32)))
    values, rhs = mesh.assemble(cu(np.ones(mesh.nE)), 1.0, cu(np.ones(mesh.nF)))
    P = ph.Schwarz(mesh, values)

    def schwarz():
        x, _, _, code = P.solve(values, rhs, rtol=1e-10, maxit=5000, check=False)
        return x, ph.ph_status_string(code)

    def refined():
        try:
            return ph.solve_refined(mesh, values, rhs, P, tol=1e-14, inner_rtol=1e-8, maxit=5000)[0], "PH_OK"
        except ph.PHError as e:
            return None, e.name

    check(ph, schwarz)
    check(ph, refined)
    P.close()
    mesh.close()
