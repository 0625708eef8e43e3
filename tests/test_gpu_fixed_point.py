"""Meshes whose elements the fixed-point geometry leaves to fp64 in whole or in
part -- stretched along an axis past its factor of 16, or with a reaction term
above a quarter of the diffusion -- against the oracle, at the bars of the
regular ones: H to 1e-12 entrywise, rhs to 1e-12 of its addends, both
recoveries to 1e-12 of each element's largest value plus 8 ulp of the terms
that cancel in it, the gradient to 1e-9.  Small meshes (fp64 throughout) with
the solve, and meshes above 32,768 tets (fixed point) with a random Lambda."""
import numpy as np
import pytest

import meshgen
import oracle
from tests.test_gpu_fullsize import EPS64, U_TERM_ULPS, recovery_terms
from tests.test_gpu_parity import assert_values_close, cu, host, run_oracle

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


@pytest.mark.parametrize("stretch,lo,c", [((1, 1, 1), 1.0, 0.1), ((1, 1, 1 / 8), 1.0, 0.1), ((1, 1, 1 / 64), 1.0, 0.1),
                                          ((1 / 512, 1, 1), 1.0, 0.1), ((1, 1, 1), 1e-3, 1.0)])
def test_left_out_elements(ph, stretch, lo, c):
    coord, tet = meshgen.kuhn_cube(2)
    coord, tet, _ = meshgen.refined(coord, tet, 1)
    coord, _ = meshgen.jitter_interior(coord, tet, 0.1, seed=6)
    coord = coord * np.asarray(stretch)
    # half of the elements on each side of the rule on the reaction term where lo < 1
    a = np.where(np.arange(tet.shape[0]) % 2 == 0, lo, 1.0)
    p = meshgen.Problem("left out", coord, tet, a, c, lambda x: meshgen.sin_source(x / np.asarray(stretch)))
    m = ph.Mesh(cu(p.coord, torch.float64), cu(p.tet, torch.int32))
    f = np.asarray(p.f(host(m.faces()["face_centroid"])))
    fd, ad = cu(f, torch.float64), cu(a, torch.float64)
    values, rhs, factor = m.assemble(ad, c, fd, factor=True)
    o = run_oracle(p)
    assert_values_close({"values": host(values), "rhs": host(rhs)}, o)
    lam, _, P = ph.solve_system(m, values, rhs, rtol=1e-13, maxit=50000)
    P.close()
    Uo = oracle.recover(p.coord, p.tet, o["fc"], o["csr"]["face_mult"], a, c, o["f"], host(lam), None)
    terms = recovery_terms(p, {"fc": o["fc"], "f": o["f"], "gN": None, "lam": host(lam), "csr": o["csr"]})
    bar = 1e-12 * np.abs(Uo).max(axis=1) + U_TERM_ULPS * EPS64 * terms
    for u in (m.recover(ad, c, fd, lam), m.recover_factored(factor, c, fd, lam)):
        assert np.all(np.abs(host(u) - Uo).max(axis=1) <= bar)
    U_obs = Uo * 1.01 + 0.01
    theta = torch.log(ad).requires_grad_(True)
    J = ph.misfit(theta, m, c, fd, cu(U_obs, torch.float64), rtol=1e-13)
    J.backward()
    J_o, g_o, _, _ = oracle.adjoint_gradient(p.coord, p.tet, a, c, p.f, U_obs)
    assert abs(J.item() - J_o) <= 1e-9 * abs(J_o)
    assert np.linalg.norm(host(theta.grad) - g_o) <= 1e-9 * np.linalg.norm(g_o)
    m.close()


def large(name):
    """Meshes above the 32,768 tets from which the record and the recovery are in fixed point."""
    if name == "mixed":
        return meshgen.problem("paper_mixed", 4)  # 103,680 tets, Neumann rows
    stretch = np.asarray({"regular": (1, 1, 1), "flat": (1, 1, 1 / 8), "left out": (1, 1 / 64, 1)}[name])
    coord, tet = meshgen.kuhn_cube(18)  # 34,992 tets
    coord, _ = meshgen.jitter_interior(coord, tet, 0.1, seed=8)
    # reaction against diffusion on both sides of the kernel's rule
    a = np.exp(np.random.default_rng(9).uniform(np.log(1e-4), np.log(1e2), tet.shape[0]))
    return meshgen.Problem(name, coord * stretch, tet, a, 1.0, lambda x: meshgen.sin_source(x / stretch))


@pytest.mark.parametrize("name", ["mixed", "regular", "flat", "left out"])
def test_large_meshes(ph, name):
    """H, rhs and both recoveries from a random Lambda; the batch gives the plain calls' bits."""
    p = large(name)
    nb = None if p.neumann is None or p.neumann.size == 0 else cu(p.neumann, torch.int32)
    m = ph.Mesh(cu(p.coord, torch.float64), cu(p.tet, torch.int32), nb)
    assert m.nE >= 32768
    o = run_oracle(p)
    f, uD, gN = (None if x is None else cu(x, torch.float64) for x in (o["f"], o["uD"], o["gN"]))
    a = cu(p.a, torch.float64)
    values, rhs, factor = m.assemble(a, p.c, f, uD_face=uD, gN_face=gN, factor=True)
    assert_values_close({"values": host(values), "rhs": host(rhs)}, o)
    lam = np.random.default_rng(10).standard_normal(m.L)
    lam_d = cu(lam, torch.float64)
    Uo = oracle.recover(p.coord, p.tet, o["fc"], o["csr"]["face_mult"], p.a, p.c, o["f"], lam, o["gN"])
    terms = recovery_terms(p, {"fc": o["fc"], "f": o["f"], "gN": o["gN"], "lam": lam, "csr": o["csr"]})
    bar = 1e-12 * np.abs(Uo).max(axis=1) + U_TERM_ULPS * EPS64 * terms
    u = m.recover_factored(factor, p.c, f, lam_d, gN)
    for w in (m.recover(a, p.c, f, lam_d, gN), u):
        assert np.all(np.abs(host(w) - Uo).max(axis=1) <= bar)
    out = [torch.full_like(x, float("nan")) for x in (values, rhs, factor, u)]
    b = ph.Batch([m])
    b.bind([a], [p.c], [f], [out[0]], [out[1]], factor=[out[2]], uD_face=[uD], gN_face=[gN])
    b.bind_recovery([lam_d], [out[3]])
    b.graph_launch()
    torch.cuda.synchronize()
    for x, y in zip(out, (values, rhs, factor, u)):
        assert torch.equal(x, y)
    b.close()
    m.close()
