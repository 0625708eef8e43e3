"""The gradient on a graded mesh above the 32,768 tets from which G_e is held in
fixed point: elements with short edges and small faces of 1 to 1/30 of the rest,
against the formula grad_T = -a p' K U, p = A^-1 (M e + C' q), in long double."""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LF = [(0, 1, 2), (0, 2, 3), (0, 3, 1), (3, 2, 1)]


def cu(x, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dt, device="cuda")


def solve4(A, b):
    """A x = b for stacks of 4x4 positive definite matrices, by elimination."""
    A, b = A.copy(), b.copy()
    for k in range(4):
        for i in range(k + 1, 4):
            w = A[:, i, k] / A[:, k, k]
            A[:, i] -= w[:, None] * A[:, k]
            b[:, i] -= w * b[:, k]
    x = np.zeros_like(b)
    for k in (3, 2, 1, 0):
        x[:, k] = (b[:, k] - sum(A[:, k, j] * x[:, j] for j in range(k + 1, 4))) / A[:, k, k]
    return x


@pytest.mark.parametrize("power", [1.0, 2.5])
def test_gradient(power):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    coord, tet = meshgen.kuhn_cube(18)
    coord, _ = meshgen.jitter_interior(coord, tet, 0.1, seed=3)
    coord = coord ** power
    rng = np.random.default_rng(4)
    nE, c = tet.shape[0], 0.1
    a = np.exp(rng.standard_normal(nE))
    m = ph.Mesh(cu(coord), cu(tet, torch.int32))
    assert m.nE >= 32768
    fc = {k: v.cpu().numpy() for k, v in m.faces().items()}
    U, Uo, q = rng.standard_normal((nE, 4)), rng.standard_normal((nE, 4)), rng.standard_normal(m.L)
    _, _, factor = m.assemble(cu(a), c, cu(np.ones(m.nF)), factor=True)
    g = m.adjoint_grad(cu(a), factor, c, cu(U), cu(Uo), cu(q)).cpu().numpy()

    P = coord.astype(np.longdouble)[tet]
    E = P[:, 1:] - P[:, :1]
    cof = np.cross(E[:, [1, 2, 0]], E[:, [2, 0, 1]])
    det = (E[:, 0] * cof[:, 0]).sum(-1)
    grads = np.concatenate([-cof.sum(1, keepdims=True), cof], axis=1) / det[:, None, None]  # of the vertex functions
    vol = np.abs(det) / 6
    K = vol[:, None, None] * np.einsum("tid,tjd->tij", grads, grads)
    M = vol[:, None, None] / 20 * (np.ones((4, 4)) + np.eye(4))
    b = np.einsum("tij,tj->ti", M, (U - Uo).astype(np.longdouble))
    F = fc["tet_face"].astype(np.int64) & 0x7FFFFFFF
    sign = np.where(fc["tet_face"].astype(np.int64) & 0x80000000, -1, 1)
    for k in range(4):
        x, y, z = (P[:, v] for v in LF[k])
        area = np.sqrt((np.cross(z - x, y - x) ** 2).sum(-1)) / 2
        l = fc["face_mult"][F[:, k]]
        for v in LF[k]:
            b[:, v] += np.where(l >= 0, sign[:, k] * area / 3 * q[l], 0)
    p = solve4(a[:, None, None] * K + c * M, b)
    ref = -a * np.einsum("ti,tij,tj->t", p, K, U)
    terms = a * np.einsum("ti,tij,tj->t", np.abs(p), np.abs(K), np.abs(U))
    # each of the formula's terms to 1e-12, as the entries of H and the recovery
    assert np.all(np.abs(g - ref) <= 1e-12 * terms)
    m.close()
