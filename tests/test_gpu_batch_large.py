"""A batch whose problems take different paths: one above the 32,768 tets from
which the element algebra runs in fixed point, between smaller ones (one with
Neumann faces), built together and alone: the same bits from the batched build
and the batched kernels, with every block shape, as from the plain calls."""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def cu(x, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=dt, device="cuda")


def problems():
    out = [meshgen.problem("paper_mixed", 2)]
    coord, tet = meshgen.kuhn_cube(18)  # 34,992 tets, some of them graded
    coord, _ = meshgen.jitter_interior(coord, tet, 0.2, seed=12)
    out.append(meshgen.Problem("large", coord * [1, 1, 0.15], tet, meshgen.lognormal_field(tet.shape[0], 13), 0.3,
                               lambda x: meshgen.sin_source(x)))
    coord, tet = meshgen.kuhn_cube(4)
    out.append(meshgen.Problem("small", coord, tet, meshgen.lognormal_field(tet.shape[0], 14), 0.3,
                               lambda x: meshgen.sin_source(x)))
    return out


def test_build_and_kernels():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    from paper_2509_11133_gb300 import build
    build.build()
    ph.load()
    ps = problems()
    arr = [(cu(p.coord), cu(p.tet, torch.int32), cu(p.neumann, torch.int32) if p.neumann.size else None) for p in ps]
    together = ph.create_meshes(*(list(x) for x in zip(*arr)))
    ref, data = [], []
    for p, x, m in zip(ps, arr, together):
        alone = ph.Mesh(*x)
        cen = alone.faces()["face_centroid"].cpu().numpy()
        f, uD, gN = (None if g is None else cu(np.asarray(g(cen))) for g in (p.f, p.uD, p.gN))
        a, lam = cu(p.a), cu(np.random.default_rng(15).standard_normal(alone.L))
        data.append((a, p.c, f, uD, gN, lam))
        outs = []
        for q in (alone, m):
            values, rhs, factor = q.assemble(a, p.c, f, uD, gN, factor=True)
            outs.append((values, rhs, factor, q.recover_factored(factor, p.c, f, lam, gN),
                         q.recover(a, p.c, f, lam, gN)))
        for s, t in zip(*outs):
            assert torch.equal(s, t)
        ref.append(outs[0])
        alone.close()
    assert [m.nE >= 32768 for m in together] == [False, True, False]
    out = [[torch.empty_like(t) for t in r[:4]] for r in ref]
    b = ph.Batch(together)
    b.bind([d[0] for d in data], [d[1] for d in data], [d[2] for d in data], [o[0] for o in out], [o[1] for o in out],
           factor=[o[2] for o in out], uD_face=[d[3] for d in data], gN_face=[d[4] for d in data])
    b.bind_recovery([d[5] for d in data], [o[3] for o in out])
    for config in ((1024, 256, 6), (96, 64, 2), (1024, 288, 2), (4096, 512, 3), (1000, 1024, 1)):
        b.set_config(*config)
        for o in out:
            for t in o:
                t.fill_(np.nan)
        b.graph_launch()
        torch.cuda.synchronize()
        for o, r in zip(out, ref):
            for s, t in zip(o, r):
                assert torch.equal(s, t)
    b.close()
    for m in together:
        m.close()


def test_autotune_times_the_present_configuration():
    """Every candidate (4 tiles, 3 thread counts, 4 blocks per SM) and the one in
    use, which need not be among them, are timed: two launches, warm-up and reps."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2509_11133_gb300 as ph
    ph.load()
    coord, tet = meshgen.kuhn_cube(4)
    m = ph.Mesh(cu(coord), cu(tet, torch.int32))
    new = lambda n: torch.zeros(n, dtype=torch.float64, device="cuda")
    b = ph.Batch([m])
    b.bind([cu(np.ones(m.nE))], [1.0], [cu(np.ones(m.nF))], [new(m.nnz)], [new(m.L)])
    b.set_config(777, 96, 5)
    before = ph.ph_launch_count()
    ms = b.autotune(reps=2)
    assert ph.ph_launch_count() - before == 2 * (1 + 2) * (4 * 3 * 4 + 1)
    assert ms > 0.0 and b.get_config()["threads"] in (64, 96, 128, 256)
    b.close()
    m.close()
