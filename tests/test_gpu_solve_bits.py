"""The one-launch conjugate gradients against the per-iteration kernels that they
replace, with the same x: the same solution, iteration count and residual, bit
for bit, with either preconditioner, at the sizes where the layout of the loop
changes (64-, 128-, 192- and 256-row blocks up to 38,912 rows, 512-row slots
above, one or more slots to a block) and with odd numbers of rows."""
import numpy as np
import pytest

import meshgen
from tests.test_gpu_solve_loop import banded_spd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


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


def cu(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def both(ph, solve):
    out = []
    for mode in (0, 1):
        ph.ph_test_pcg_loop(mode)
        before = ph.ph_launch_count()
        x, it, rr = solve()[:3]
        out.append((x.clone(), it, rr, ph.ph_launch_count() - before))
    ph.ph_test_pcg_loop(0)
    assert out[0][3] < 8 < out[1][3]  # the two routes were taken
    assert torch.equal(out[0][0], out[1][0]) and out[0][1:3] == out[1][1:3]
    return out[0]


@pytest.mark.parametrize("n", [1, 2, 63, 65, 9729, 19457, 29183, 38911, 38912, 38913, 77825, 155647, 233473, 311295, 311296])
@pytest.mark.parametrize("offsets", [(1, 7, 50), (1, 2, 3, 5, 9, 17, 33, 65, 129, 257)])
def test_jacobi(ph, n, offsets):
    if len(offsets) > 3 and n not in (65, 9729, 38913):
        pytest.skip("rows wider than the ELL copy: one size of each layout")
    A = banded_spd(n, offsets, n)
    b = np.random.default_rng(n + 1).standard_normal(n)
    rp, ci, va, bd = cu(A.indptr.astype(np.int32)), cu(A.indices.astype(np.int32)), cu(A.data), cu(b)
    _, it, _, _ = both(ph, lambda: ph.ph_solve_pcg(rp, ci, va, bd, rtol=1e-12, maxit=5000))
    assert it > 0
    if n <= ph.PH_PCG_NOALLOC_MAX_N:
        both(ph, lambda: ph.ph_solve_pcg_noalloc(rp, ci, va, bd, rtol=1e-12, maxit=5000))


# rows: 12 m^3 + 6 m^2, less the Neumann faces (an odd number of them)
@pytest.mark.parametrize("m,neumann", [(2, 0), (2, 3), (7, 1), (14, 0), (14, 5), (15, 1), (18, 7), (29, 3)])
def test_schwarz(ph, m, neumann):
    coord, tet = meshgen.kuhn_cube(m)
    coord, _ = meshgen.jitter_interior(coord, tet, 0.1, seed=m)
    rng = np.random.default_rng(m)
    top = [f for f in _boundary(tet) if np.all(coord[list(f), 2] == 1.0)][:neumann]
    nb = cu(np.array(top, np.int32)) if neumann else None
    mesh = ph.Mesh(cu(coord), cu(tet.astype(np.int32)), nb)
    assert mesh.L == 12 * m ** 3 + 6 * m ** 2 - neumann
    a = cu(np.exp(rng.standard_normal(mesh.nE)))
    gN = cu(np.ones(mesh.nF)) if neumann else None
    values, rhs = mesh.assemble(a, 0.1, cu(np.ones(mesh.nF)), None, gN)
    P = ph.Schwarz(mesh, values)
    rtol, maxit = (1e-10, 400) if m < 20 else (1e-10, 40)
    _, it, _, _ = both(ph, lambda: P.solve(values, rhs, rtol=rtol, maxit=maxit, check=False))
    assert it > 0
    P.close()
    mesh.close()


def _boundary(tet):
    faces = np.concatenate([tet[:, f] for f in ([0, 1, 2], [0, 2, 3], [0, 3, 1], [3, 2, 1])])
    _, inv, cnt = np.unique(np.sort(faces, axis=1), axis=0, return_inverse=True, return_counts=True)
    return [tuple(f) for f in faces[cnt[inv.ravel()] == 1]]
