"""The two builds of a mesh, by one block (up to 1,536 tets) and by the general
kernels: a mesh with two faults reports the same one from both (invalid ids
before degenerate tets before faces that do not match), and both can be timed."""
import numpy as np
import pytest

import meshgen
import oracle
from tests.test_gpu_parity import cu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 6, 7])  # 48, 1,296 and 2,058 tets
def test_first_fault(m):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    coord, tet = meshgen.kuhn_cube(m)
    flat = coord.copy()
    flat[tet[5, 3]] = flat[tet[5, 2]]  # a tet without volume
    fc = oracle.faces(tet, coord.shape[0], None)
    inner = fc["face_vtx"][fc["face_tet"][:, 1] >= 0][:1].astype(np.int32)
    thrice = np.vstack([tet, tet[:1], tet[:1]])
    wrong = tet.copy()
    wrong[3, 1] = coord.shape[0]

    def code(x, t, nb=None):
        with pytest.raises(ph.PHError) as e:
            ph.Mesh(cu(x, torch.float64), cu(t, torch.int32), None if nb is None else cu(nb, torch.int32))
        return e.value.name

    assert code(coord, thrice) == "PH_ERR_NONMANIFOLD"
    assert code(coord, tet, inner) == "PH_ERR_ARG"
    assert code(flat, tet) == "PH_ERR_DEGENERATE"
    assert code(flat, thrice) == "PH_ERR_DEGENERATE"
    assert code(flat, tet, inner) == "PH_ERR_DEGENERATE"
    assert code(flat, wrong) == "PH_ERR_ARG"
    assert code(flat, np.vstack([wrong, thrice])) == "PH_ERR_ARG"
    ph.Mesh(cu(coord, torch.float64), cu(tet, torch.int32)).close()


@pytest.mark.parametrize("m,kernels", [(6, ("k_small_connect", "k_small_geom")), (7, ("k_face_fill", "k_row_fill"))])
def test_build_kernels_are_timed(m, kernels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    ph.load()
    coord, tet = meshgen.kuhn_cube(m)
    for k in kernels:
        ph.ph_kernel_time(k, reset=True)
    ph.ph_timing_enable(2)
    try:
        ph.Mesh(cu(coord, torch.float64), cu(tet, torch.int32)).close()
    finally:
        ph.ph_timing_enable(0)
    for k in kernels:
        ms, n = ph.ph_kernel_time(k, reset=True)
        assert n == 1 and ms > 0.0
