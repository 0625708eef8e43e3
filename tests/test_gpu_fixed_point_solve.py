"""Solves of a system above the 32,768 tets from which H is formed in fixed point,
with either preconditioner, against the oracle's system and its solution.

The residual of the oracle's system (in binary128) is at most what the solver
stops at, rtol |b|, and what rounding adds to it: the entries of both systems
(within 2 x 2^-53 x 8 of each other, the parity tests' order) and one rounding per
iteration of the recurrences, (iterations + 16) 2^-53 of | |H||x| + |b| |.  The
error is then at most that over the smallest eigenvalue of H (found by inverse
iteration, to 10%)."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spla

import meshgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
RTOL = 1e-11


def cu(x, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dt, device="cuda")


@pytest.fixture(scope="module")
def system():
    coord, tet = meshgen.kuhn_cube(18)  # 34,992 tets
    coord, _ = meshgen.jitter_interior(coord, tet, 0.1, seed=8)
    p = meshgen.Problem("solve", coord, tet, meshgen.lognormal_field(tet.shape[0], 21), 1.0,
                        lambda x: meshgen.sin_source(x))
    o = oracle.pipeline(p.coord, p.tet, p.a, p.c, p.f, do_solve=False)
    L, csr = o["csr"]["L"], o["csr"]
    H = sp.csr_matrix((o["values"], csr["colind"], csr["rowptr"]), shape=(L, L))
    lu = spla.splu(H.tocsc())
    residual = lambda x: oracle.residual(csr["rowptr"], csr["colind"], o["values"], x, o["rhs"])
    x = lu.solve(o["rhs"])
    for _ in range(3):
        x += lu.solve(residual(x))
    v = np.random.default_rng(1).standard_normal(L)
    for _ in range(30):
        w = lu.solve(v)
        least = np.linalg.norm(v) / np.linalg.norm(w)
        v = w / np.linalg.norm(w)
    return p, o, H, residual, x, 0.9 * least


@pytest.mark.parametrize("precond", ["jacobi", "schwarz"])
def test_solution(system, precond):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    p, o, H, residual, exact, least = system
    m = ph.Mesh(cu(p.coord), cu(p.tet, torch.int32))
    assert m.nE >= 32768
    values, rhs = m.assemble(cu(p.a), p.c, cu(o["f_face"]))
    lam, it, P = ph.solve_system(m, values, rhs, RTOL, 20000, precond)
    if P is not None:
        P.close()
    m.close()
    lam = lam.cpu().numpy()
    b = o["rhs"]
    bound = RTOL * np.linalg.norm(b) + (it + 16) * 2.0 ** -53 * np.linalg.norm(abs(H) @ np.abs(lam) + np.abs(b))
    assert np.linalg.norm(residual(lam)) <= bound
    assert np.linalg.norm(lam - exact) <= bound / least
