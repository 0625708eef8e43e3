"""Meshes around the size up to which the connectivity is built by one block
(1,536 tets), around its 1,024 threads, and the smallest, with and without
Neumann faces: faces, signs, multipliers and the CSR pattern equal to the
oracle's, assembly at the parity bars; invalid small meshes refused."""
import numpy as np
import pytest

import meshgen
import oracle
from tests.test_gpu_parity import cu, host

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
    return ph


def part(n, shuffle):
    coord, tet = meshgen.kuhn_cube(4)
    coord, tet, _ = meshgen.refined(coord, tet, 1)
    if shuffle:
        coord, tet = meshgen.shuffled(coord, tet, 5)
    tet = tet[:n]
    used, ids = np.unique(tet, return_inverse=True)  # the part's own vertices
    return coord[used], ids.reshape(-1, 4).astype(np.int32)


@pytest.mark.parametrize("n", [1, 2, 33, 511, 1023, 1024, 1025, 1535, 1536, 1537])
@pytest.mark.parametrize("neumann", [False, True])
@pytest.mark.parametrize("shuffle", [False, True])
def test_small_mesh_against_oracle(ph, n, neumann, shuffle):
    coord, tet = part(n, shuffle)
    fc = oracle.faces(tet, coord.shape[0], None)
    nb = None
    if neumann:  # every third boundary face, in another order than the faces'
        nb = fc["face_vtx"][fc["face_tet"][:, 1] < 0][::-3][:, [1, 2, 0]].astype(np.int32)
        fc = oracle.faces(tet, coord.shape[0], nb)
    fm, L = oracle.multipliers(fc["face_kind"])
    rp, ci = oracle.csr_pattern(fc["tet_face"], fm, L)
    m = ph.Mesh(cu(coord, torch.float64), cu(tet, torch.int32), None if nb is None else cu(nb, torch.int32))
    g = {k: host(v) for k, v in m.faces().items()}
    rowptr, colind = m.csr_pattern()
    for k in ("tet_face", "face_tet", "face_vtx", "face_kind"):
        assert np.array_equal(g[k], fc[k]), k
    assert np.array_equal(g["face_mult"], fm) and m.L == L
    assert np.array_equal(host(rowptr), rp) and np.array_equal(host(colind), ci)
    a = np.random.default_rng(n).uniform(0.5, 2.0, n)
    cen = g["face_centroid"]
    f = meshgen.sin_source(cen)
    gN = None if nb is None else 1.0 + cen[:, 0]
    values, rhs = m.assemble(cu(a, torch.float64), 0.7, cu(f, torch.float64),
                             gN_face=None if gN is None else cu(gN, torch.float64))
    v, r, mag = oracle.assemble(coord, tet, fc, {"face_mult": fm, "L": L, "rowptr": rp, "colind": ci}, a, 0.7, f, None, gN)
    assert np.all(np.abs(host(values) - v) <= 1e-12 * np.abs(v))
    assert np.all(np.abs(host(rhs) - r) <= 1e-12 * mag + 1e-300)
    m.close()


def test_small_invalid_meshes(ph):
    coord, tet = part(100, False)
    c = cu(coord, torch.float64)

    def code(t, nb=None, x=c):
        with pytest.raises(ph.PHError) as e:
            ph.Mesh(x, cu(t, torch.int32), None if nb is None else cu(nb, torch.int32))
        return e.value.name

    bad = tet.copy()
    bad[7, 2] = coord.shape[0]
    assert code(bad) == "PH_ERR_ARG"
    bad = tet.copy()
    bad[7, 2] = bad[7, 1]
    assert code(bad) == "PH_ERR_ARG"
    assert code(np.vstack([tet, tet[:1], tet[:1]])) == "PH_ERR_NONMANIFOLD"
    fc = oracle.faces(tet, coord.shape[0], None)
    inner = fc["face_vtx"][fc["face_tet"][:, 1] >= 0][:1].astype(np.int32)
    outer = fc["face_vtx"][fc["face_tet"][:, 1] < 0][:1].astype(np.int32)
    assert code(tet, inner) == "PH_ERR_ARG"
    assert code(tet, np.vstack([outer, outer])) == "PH_ERR_ARG"
    flat = coord.copy()
    flat[:, 2] = 0.0
    assert code(tet, x=cu(flat, torch.float64)) == "PH_ERR_DEGENERATE"
    ph.Mesh(c, cu(tet, torch.int32)).close()
