"""Performance cases of the primal hybrid FEM library: the work a user's
program has it do, through the public Python entry points, over the range of
sizes, meshes, boundary conditions and options the library is used with.

Kinds of pass (``case["kind"]``):

- ``step``: mesh build, assembly with the element factor and recovery from
  given face values (the data-parallel path; the solve is done elsewhere);
- ``forward``: mesh build, assembly, solve and recovery of one problem;
- ``gradient``: misfit and its gradient in log a on a mesh that the program
  keeps (one step of an inversion);
- ``refine``: a chain of uniform refinements with the boundary lists;
- ``batch``: many problems of uneven size, from their vertices to the
  recovered values (``build`` true) or the kept batch's graph (false);
- ``host``: the path from and to page-locked host buffers.

Meshes are the Listing-1 five-tet cube or the Kuhn m^3 cube, refined
``levels`` times; ``jitter`` moves the interior vertices, ``shuffle`` renumbers
vertices and tets at random.  The coefficient is 1, lognormal, or 1/1e4 on an
8^3 checkerboard; the boundary is Dirichlet, or mixed (Dirichlet on z = 1 only).
"""
import math

import numpy as np
import torch

import paper_2509_11133_gb300 as ph

FACES = [[0, 1, 2], [0, 2, 3], [0, 3, 1], [3, 2, 1]]  # local faces; face k lies opposite vertex OPP[k]
OPP = [3, 1, 2, 0]
EDGES = [[0, 1], [0, 2], [0, 3], [1, 2], [1, 3], [2, 3]]  # local edges IJ, IK, IL, JK, JL, KL
DENSE_MAX = 24000  # unknowns up to which exact() solves the system (dense Cholesky)


def _case(name, kind, m, levels, **more):
    c = {"name": name, "kind": kind, "mesh": "kuhn", "m": m, "levels": levels, "jitter": 0.0, "shuffle": False,
         "field": "lognormal", "c": 0.1, "boundary": "dirichlet", "variant": "f64"}
    c.update(more)
    return c


def listed():
    return [
        # the paper's own example (Listing 1, mixed conditions) at level 2: the smallest whole solve, bound by latency
        _case("forward_mixed_720", "forward", 1, 2, mesh="cube5", field="one", c=1.0, boundary="mixed",
              solver="schwarz", rtol=1e-12),
        # the smallest configuration (864 tets): mesh, system and recovery, bound by launches
        _case("step_sin_864", "step", 1, 2, field="one", c=1.0, pattern=True),
        # an ordinary mesh of a few million tets with a random coefficient
        _case("step_lognormal_3m", "step", 3, 4),
        # the largest configuration: 17.9M jittered tets, coefficient contrast 1e4
        _case("step_jitter_checker_18m", "step", 1, 6, jitter=0.2, field="checker", c=1.0),
        # the double-word precision variant on its own mesh record
        _case("step_dw_lognormal_1m", "step", 2, 4, variant="dw"),
        # a mesh as an unstructured generator numbers it (no locality), Neumann rows, pattern read out
        _case("step_shuffled_mixed_296k", "step", 7, 2, shuffle=True, boundary="mixed", pattern=True),
        # growing a mesh on the device from the coarse cube, boundary lists along
        _case("refine_12m", "refine", 2, 5, boundary="mixed"),
        # one problem with the plain Jacobi solver (thousands of cheap iterations)
        _case("forward_jacobi_23k", "forward", 3, 2, solver="jacobi", rtol=1e-10),
        # an ill-conditioned problem solved to fp64 accuracy
        _case("forward_refined_10k", "forward", 1, 3, jitter=0.2, field="checker", c=1.0, solver="refined"),
        # one inversion step on the adjoint configuration
        _case("gradient_2m", "gradient", 6, 3, rtol=1e-10),
        # the batched configuration: 256 problems of 1e4 to 5e5 tets
        _case("batch_256", "batch", 0, 1, problems=256, lo=1e4, hi=5e5, sizes_seed=4, build=True),
        # a caller with host memory only
        _case("host_lognormal_1m", "host", 2, 4),
    ]


def _pick_mesh(rng, lo, hi, max_levels=5):
    """(mesh, m, levels) with a tet count log-uniform in about [lo, hi]."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.15:
        return "cube5", 1, max(0, min(max_levels, round(math.log(target / 5) / math.log(12))))
    levels = rng.randint(0, max(0, min(max_levels, int(math.log(max(target, 6) / 6) / math.log(12)))))
    return "kuhn", max(1, round((target / (6 * 12 ** levels)) ** (1 / 3))), levels


def draw(rng):
    kind = rng.choice(["step", "step", "step", "forward", "forward", "gradient", "refine", "batch", "host"])
    more = {"c": rng.choice([0.1, 1.0, 0.01]), "boundary": rng.choice(["dirichlet", "mixed"])}
    if kind == "step":
        mesh, m, levels = _pick_mesh(rng, 60, 4e6)
        more.update(jitter=rng.choice([0.0, 0.1, 0.2]), shuffle=rng.random() < 0.25,
                    field=rng.choice(["one", "lognormal", "checker"]), variant=rng.choice(["f64", "f64", "f64", "dw"]),
                    pattern=rng.random() < 0.5)
    elif kind == "forward":
        solver = rng.choice(["schwarz", "schwarz", "jacobi", "refined"])
        mesh, m, levels = _pick_mesh(rng, 60, {"schwarz": 3e5, "jacobi": 2e4, "refined": 1e4}[solver], 3)
        more.update(solver=solver, rtol=1e-10, field=rng.choice(["one", "lognormal"]), jitter=rng.choice([0.0, 0.1]),
                    shuffle=rng.random() < 0.25)
    elif kind == "gradient":
        mesh, m, levels = _pick_mesh(rng, 500, 1e6, 3)
        more.update(rtol=1e-10)
    elif kind == "refine":
        mesh, m, levels = _pick_mesh(rng, 720, 1e7, 5)
        levels = max(1, levels)
        more.update(jitter=rng.choice([0.0, 0.2]), shuffle=rng.random() < 0.25)
        m = min(m, max(1, int((1.1e7 / (6 * 12 ** levels)) ** (1 / 3))))
    elif kind == "batch":
        mesh, m, levels = "kuhn", 0, 1
        lo = math.exp(rng.uniform(math.log(1e3), math.log(2e4)))
        more.update(problems=rng.randint(2, 96), lo=lo, hi=lo * rng.uniform(2.0, 20.0), sizes_seed=rng.randint(0, 999),
                    build=rng.random() < 0.5, boundary="dirichlet")
    else:
        mesh, m, levels = _pick_mesh(rng, 700, 3e6, 4)
        more.update(field=rng.choice(["lognormal", "checker"]), jitter=rng.choice([0.0, 0.2]))
    c = _case("", kind, m, levels, mesh=mesh, **more)
    del c["name"]
    return c


# --- inputs ------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _kuhn(m):
    """Unit cube of m^3 subcubes, each split into the 6 tets around its diagonal."""
    n = m + 1
    k, j, i = (x.ravel() for x in np.meshgrid(np.arange(n), np.arange(n), np.arange(n), indexing="ij"))
    coord = np.stack([i, j, k], axis=1) / m
    base = (np.arange(n ** 3).reshape(n, n, n)[:m, :m, :m]).ravel()
    step = (1, n, n * n)
    tets = [np.stack([base, base + step[a], base + step[a] + step[b], base + sum(step)], axis=1)
            for a in range(3) for b in range(3) if b != a]
    return coord, np.stack(tets, axis=1).reshape(-1, 4)


def _coarse(case):
    """Coarse coordinates, tets and the Neumann triples (numpy; none if Dirichlet)."""
    if case["mesh"] == "cube5":  # Listing 1
        coord = np.array([[i & 1, i >> 1 & 1, i >> 2] for i in range(8)], dtype=np.float64)
        tet = np.array([[1, 2, 3, 5], [5, 8, 6, 2], [7, 3, 8, 5], [4, 8, 3, 2], [8, 3, 2, 5]]) - 1
    else:
        coord, tet = _kuhn(case["m"])
    tri = tet[:, FACES].reshape(-1, 3)
    _, first, count = np.unique(np.sort(tri, axis=1), axis=0, return_index=True, return_counts=True)
    nb = tri[np.sort(first[count == 1])]
    nb = nb[~np.all(coord[nb][:, :, 2] == 1.0, axis=1)] if case["boundary"] == "mixed" else nb[:0]
    return coord, tet.astype(np.int32), nb.astype(np.int32)


def _cu(x):
    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _jitter(coord, tet, frac, gen):
    """Interior vertices moved within frac of their shortest edge; the vertices
    of a tet that falls below 10% of its volume move back halfway, three times,
    and then stay where they were."""
    t = tet.long()
    e = t[:, EDGES].reshape(-1, 2)
    length = (coord[e[:, 0]] - coord[e[:, 1]]).norm(dim=1)
    h = torch.full((coord.shape[0],), math.inf, dtype=torch.float64, device=coord.device)
    for j in (0, 1):
        h.scatter_reduce_(0, e[:, j], length, "amin")
    del e, length
    inner = ((coord > 0) & (coord < 1)).all(dim=1)
    d = torch.randn(coord.shape, dtype=torch.float64, device=coord.device, generator=gen)
    d *= (frac * h * inner * torch.rand(h.shape, dtype=torch.float64, device=coord.device, generator=gen) ** (1 / 3)
          / d.norm(dim=1)).unsqueeze(1)

    def volume(x):
        p = x[t]
        return ((p[:, 1] - p[:, 0]) * torch.linalg.cross(p[:, 2] - p[:, 0], p[:, 3] - p[:, 0])).sum(1)

    v0 = volume(coord)
    for scale in (0.5, 0.5, 0.5, 0.0, 0.0, 0.0):
        bad = ~(volume(coord + d) / v0 >= 0.1)
        move = torch.zeros(coord.shape[0], dtype=torch.bool, device=coord.device)
        move[t[bad].reshape(-1)] = True
        d[move] *= scale
    return (coord + d).contiguous()


def _mesh_arrays(case, gen):
    coord, tet, nb = (_cu(x) for x in _coarse(case))
    for _ in range(case["levels"]):
        coord, tet, lists, _ = ph.ph_refine(coord, tet, nb if nb.shape[0] else None)
        nb = lists if lists is not None else nb
    if case["jitter"]:
        coord = _jitter(coord, tet, case["jitter"], gen)
    if case["shuffle"]:
        new = torch.randperm(coord.shape[0], device="cuda", generator=gen)  # vertex v becomes new[v]
        moved = torch.empty_like(coord)
        moved[new] = coord
        coord, ids = moved, new.to(torch.int32)
        tet, nb = ids[tet.long()], ids[nb.long()]
        tet = tet[torch.randperm(tet.shape[0], device="cuda", generator=gen)]
        turn = torch.randint(0, 4, (tet.shape[0], 1), device="cuda", generator=gen)
        tet = tet.gather(1, (torch.arange(4, device="cuda") + turn) % 4).contiguous()
        nb = nb[torch.randperm(nb.shape[0], device="cuda", generator=gen)].contiguous()
    return coord, tet, (nb if nb.shape[0] else None)


def _field(case, coord, tet, gen):
    n = tet.shape[0]
    if case["field"] == "one":
        return torch.ones(n, dtype=torch.float64, device="cuda")
    if case["field"] == "lognormal":
        return torch.exp(torch.randn(n, dtype=torch.float64, device="cuda", generator=gen))
    block = (8 * coord[tet.long()].mean(dim=1)).floor().long().clamp(0, 7).sum(dim=1)
    return torch.where(block % 2 == 1, 1e4, 1.0).to(torch.float64)


def _sin3(x):
    return torch.sin(math.pi * x).prod(dim=-1)


def _problem(case, seed, mesh_of=None):
    """Mesh arrays, coefficient and face data of one problem; with `mesh_of`
    also the counts of its mesh (a mesh is built for its face centroids)."""
    gen = _gen(seed)
    coord, tet, nb = _mesh_arrays(case, gen)
    s = {"coord": coord, "tet": tet, "nb": nb, "a": _field(case, coord, tet, gen), "c": case["c"], "gen": gen}
    m = ph.Mesh(coord, tet, nb)
    cen = m.faces()["face_centroid"]
    amp = 0.5 + float(torch.rand((), device="cuda", generator=gen))
    s["uD"] = s["gN"] = None
    if case["boundary"] == "mixed":  # u = x^2 y^2 z^2, the paper's example
        q = cen ** 2
        s["f"] = amp * (q.prod(1) - 2 * (q[:, 1] * q[:, 2] + q[:, 0] * q[:, 2] + q[:, 0] * q[:, 1]))
        s["uD"] = amp * q.prod(1)
        grad = 2 * torch.stack([cen[:, 0] * q[:, 1] * q[:, 2], q[:, 0] * cen[:, 1] * q[:, 2],
                                q[:, 0] * q[:, 1] * cen[:, 2]], dim=1)
        normal = (cen >= 1 - 1e-12).double() - (cen <= 1e-12).double()
        s["gN"] = amp * (grad * normal).sum(1)
    else:
        s["f"] = amp * (3 * math.pi ** 2 + 1) * _sin3(cen)
    s["counts"] = (m.nF, m.L, m.nnz)
    s["mesh"] = m
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind == "refine":
        coord, tet, nb = _mesh_arrays(dict(case, levels=0), _gen(seed))
        stretch = 1 + torch.rand(3, dtype=torch.float64, device="cuda", generator=_gen(seed + 1))
        return {"case": case, "coord": coord * stretch, "tet": tet, "nb": nb}
    if kind == "batch":
        return _prepare_batch(case, seed)
    s = _problem(case, seed)
    s["case"] = case
    m = s["mesh"]
    if kind in ("step", "host"):
        s["lam"] = torch.rand(m.L, dtype=torch.float64, device="cuda", generator=s["gen"]) * 2 - 1
    if kind == "gradient":
        p = s["coord"][s["tet"].long()]
        s["u_obs"] = _sin3(p) * (1 + 0.01 * torch.randn(p.shape[:2], dtype=torch.float64, device="cuda",
                                                        generator=s["gen"]))
        s["theta"] = torch.log(s["a"])
        return s
    del s["mesh"]
    m.close()
    if kind == "host":
        for k in ("coord", "tet", "nb", "a", "f", "uD", "gN", "lam"):
            if s[k] is not None:
                s[k] = s[k].cpu().pin_memory()
        nF, L, nnz = s["counts"]
        new = lambda shape, dt: torch.empty(shape, dtype=dt, pin_memory=True)
        s["out"] = {"rowptr": new(L + 1, torch.int32), "colind": new(nnz, torch.int32),
                    "values": new(nnz, torch.float64), "rhs": new(L, torch.float64),
                    "u": new((s["tet"].shape[0], 4), torch.float64)}
    return s


def _batch_sizes(case):
    rng = np.random.Generator(np.random.PCG64(case["sizes_seed"]))
    sizes = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), case["problems"]))
    return [int(min(max(round((x / 72) ** (1 / 3)), 2), 19)) for x in sizes]


def _prepare_batch(case, seed):
    """Problems of uneven size; outputs bound to slices of four flat buffers."""
    gen = _gen(seed)
    s = {"case": case, "coord": [], "tet": [], "f": [], "a": [], "c": [case["c"]] * case["problems"]}
    sized, counts = {}, []
    for m in _batch_sizes(case):
        if m not in sized:
            coord, tet, _ = _mesh_arrays(dict(case, m=m, boundary="dirichlet"), gen)
            mesh = ph.Mesh(coord, tet)
            sized[m] = (coord, tet, mesh.faces()["face_centroid"], (mesh.L, mesh.nnz, mesh.nE))
            mesh.close()
        coord, tet, cen, n = sized[m]
        s["coord"].append(coord)
        s["tet"].append(tet.clone())
        s["a"].append(torch.exp(torch.randn(n[2], dtype=torch.float64, device="cuda", generator=gen)))
        s["f"].append((3 * math.pi ** 2 + 1) * _sin3(cen))
        counts.append(n)
    new = lambda k: torch.empty(k, dtype=torch.float64, device="cuda")
    L, nnz, nE = (sum(n[i] for n in counts) for i in range(3))
    s["flat"] = {"values": new(nnz), "rhs": new(L), "factor": new(10 * nE), "u": new(4 * nE)}
    cut = lambda k, sizes: list(torch.split(s["flat"][k], sizes))
    s["bound"] = {"values": cut("values", [n[1] for n in counts]), "rhs": cut("rhs", [n[0] for n in counts]),
                  "factor": cut("factor", [10 * n[2] for n in counts]), "u": cut("u", [4 * n[2] for n in counts])}
    s["lam"] = list(torch.split(torch.rand(L, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1,
                                [n[0] for n in counts]))
    if not case["build"]:
        s["batch"] = _batch(s)
    return s


def _batch(s):
    meshes = ph.create_meshes(s["coord"], s["tet"])
    b = ph.Batch(meshes)
    o = s["bound"]
    b.bind(s["a"], s["c"], s["f"], o["values"], o["rhs"], o["factor"])
    b.bind_recovery(s["lam"], o["u"])
    return b


# --- one pass ----------------------------------------------------------------
def run(s):
    return {"step": _run_step, "forward": _run_forward, "gradient": _run_gradient, "refine": _run_refine,
            "batch": _run_batch, "host": _run_host}[s["case"]["kind"]](s)


def _run_step(s):
    v = s["case"]["variant"]
    m = ph.Mesh(s["coord"], s["tet"], s["nb"], geometry=v)
    values, rhs, factor = m.assemble(s["a"], s["c"], s["f"], s["uD"], s["gN"], factor=True, variant=v)
    u = m.recover_factored(factor, s["c"], s["f"], s["lam"], s["gN"], variant=v)
    out = {"values": values, "rhs": rhs, "factor": factor, "u": u}
    if s["case"].get("pattern"):
        out["rowptr"], out["colind"] = m.csr_pattern()
    m.close()
    return out


def _run_forward(s):
    case = s["case"]
    m = ph.Mesh(s["coord"], s["tet"], s["nb"])
    values, rhs = m.assemble(s["a"], s["c"], s["f"], s["uD"], s["gN"])
    if case["solver"] == "refined":
        P = ph.Schwarz(m, values)
        lam = ph.solve_refined(m, values, rhs, P, tol=1e-15, inner_rtol=1e-8, maxit=200000)[0]
    else:
        lam, _, P = ph.solve_system(m, values, rhs, rtol=case["rtol"], maxit=200000, precond=case["solver"])
    u = m.recover(s["a"], s["c"], s["f"], lam, s["gN"])
    if P is not None:
        P.close()
    m.close()
    return {"values": values, "rhs": rhs, "lam": lam, "u": u}


def _run_gradient(s):
    theta = s["theta"].detach().requires_grad_(True)
    J = ph.misfit(theta, s["mesh"], s["c"], s["f"], s["u_obs"], s["uD"], s["gN"], rtol=s["case"]["rtol"])
    J.backward()
    return {"J": J.detach(), "grad": theta.grad}


def _run_refine(s):
    coord, tet, nb = s["coord"], s["tet"], s["nb"]
    for _ in range(s["case"]["levels"]):
        coord, tet, nb, _ = ph.ph_refine(coord, tet, nb)
    out = {"coord": coord, "tet": tet}
    if nb is not None:
        out["neumann"] = nb
    return out


def _run_batch(s):
    if s["case"]["build"]:
        b = _batch(s)
        b.assemble()
        b.close()
        for m in b.meshes:
            m.close()
    else:
        s["batch"].graph_launch()
    return dict(s["flat"])


def _run_host(s):
    return ph.ph_assemble_host(s["coord"], s["tet"], s["a"], s["c"], s["f"], s["counts"], lam=s["lam"],
                               uD_face=s["uD"], gN_face=s["gN"], neumann=s["nb"], out=s["out"])


# --- the work a pass cannot do without ----------------------------------------
def _counts(case):
    """(nC, nE, nF, L, nnz) of a case's mesh, and its Neumann faces, from Euler's
    formula nC - nEd + nF - nE = 1 and the refinement's recursions."""
    m, k = case["m"], case["levels"]
    nE, nC, nB = (5, 8, 12) if case["mesh"] == "cube5" else (6 * m ** 3, (m + 1) ** 3, 12 * m * m)
    for _ in range(k):
        nC += nE + (nC + (4 * nE + nB) // 2 - nE - 1)
        nE, nB = 12 * nE, 4 * nB
    nF = (4 * nE + nB) // 2
    nN = nB * 5 // 6 if case["boundary"] == "mixed" else 0
    # a row has 1 + 3 entries per tet of its face, a Neumann face takes its row and its 3 columns out
    return nC, nE, nF, nF - nN, nF + 12 * nE - 7 * nN, nN


def _step_work(case):
    nC, nE, nF, L, nnz, nN = _counts(case)
    b = 24 * nC + 16 * nE + 12 * nN + 8 * nE + 8 * nF + 8 * L + 8 * nnz + 8 * L + 32 * nE
    b += 16 * nF * (case["boundary"] == "mixed")
    if case["kind"] in ("step", "batch"):
        b += 80 * nE
    if case.get("pattern") or case["kind"] == "host":
        b += 4 * (L + 1) + 4 * nnz
    return b, 360 * nE, nE, L, nnz  # flops: the element formulas, two per fused multiply-add


def work(case):
    kind = case["kind"]
    if kind == "refine":
        nC0, nE0 = _counts(dict(case, levels=0))[:2]
        nC, nE, _, _, _, nN = _counts(case)
        return {"bytes": 24 * (nC0 + nC) + 16 * (nE0 + nE) + 13 * nN, "flops": 6 * nC}
    if kind == "batch":
        per = [_step_work(dict(case, m=m)) for m in _batch_sizes(case)]
        return {"bytes": sum(p[0] for p in per), "flops": sum(p[1] for p in per)}
    b, flops, nE, L, nnz = _step_work(case)
    if kind == "forward":
        flops += 2 * nnz
    if kind == "gradient":
        return {"bytes": 2 * (12 * nnz + 16 * L) + 32 * nE + 24 * nE, "flops": 2 * flops + 4 * nnz}
    return {"bytes": b, "flops": flops}


# --- the same in plain torch, 64 bits ------------------------------------------
def _first_rank(inv):
    """Ids by first occurrence, and the first slot, of each slot's class."""
    n = int(inv.max()) + 1 if inv.numel() else 0
    slot = torch.arange(inv.numel(), device=inv.device)
    first = torch.full((n,), inv.numel(), dtype=torch.int64, device=inv.device).scatter_reduce_(0, inv, slot, "amin")
    rank = torch.empty_like(first)
    rank[first.argsort()] = torch.arange(n, device=inv.device)
    return rank[inv], first[inv]


def _triple_classes(tri, nC):
    tri = tri.long().sort(dim=1).values
    _, pair = torch.unique(tri[:, 1] * nC + tri[:, 2], return_inverse=True)
    return torch.unique(pair * nC + tri[:, 0], return_inverse=True)[1]


def _exact_system(coord, tet, nb, a, c, f, uD, gN):
    """The condensed system by its definition; A^-1 = J/(c|T|) + X (a I + c/20 X'X)^-1 X'/|T|
    on the vertex positions X about the centroid
    (from the edge vectors, whose rounding is relative to the element's size)."""
    nE, nC = tet.shape[0], coord.shape[0]
    tri = tet[:, FACES].reshape(-1, 3)
    fid, first = _first_rank(_triple_classes(tri if nb is None else torch.cat([tri, nb]), nC))
    neu = fid[4 * nE:]
    fid, first = fid[:4 * nE], first[:4 * nE]
    nF = int(fid.max()) + 1
    owner = torch.zeros(nF, dtype=torch.int64, device=coord.device)
    slot = torch.arange(4 * nE, device=coord.device)
    owner[fid] = first
    p = coord[tri[owner].long()]
    area = 0.5 * torch.linalg.cross(p[:, 2] - p[:, 0], p[:, 1] - p[:, 0]).norm(dim=1)
    has = torch.ones(nF, dtype=torch.bool, device=coord.device)
    has[neu] = False
    mult = torch.cumsum(has, 0) - 1
    L = int(has.sum())
    P = coord[tet.long()]
    E = P[:, 1:] - P[:, :1]
    vol = (E[:, 0] * torch.linalg.cross(E[:, 1], E[:, 2])).sum(1).abs() / 6
    X = torch.cat([torch.zeros_like(E[:, :1]), E], dim=1)
    X = X - X.mean(dim=1, keepdim=True)
    M = (c / 20) * X.transpose(1, 2) @ X
    M.diagonal(dim1=1, dim2=2).add_(a[:, None])
    r0, r1, r2 = M.unbind(1)
    cof = torch.stack([torch.linalg.cross(r1, r2), torch.linalg.cross(r2, r0), torch.linalg.cross(r0, r1)], dim=1)
    cof /= (r0 * cof[:, 0]).sum(1)[:, None, None]
    Q = X @ (cof @ X.transpose(1, 2)) / vol[:, None, None]
    Q = Q[:, OPP][:, :, OPP]  # face-indexed
    fid4 = fid.view(nE, 4)
    sgn = torch.where(slot == first, 1.0, -1.0).double().view(nE, 4)
    d = sgn * area[fid4]
    h = vol[:, None] / 4 * f[fid4]
    if gN is not None:
        h = h + torch.where(has[fid4], 0.0, area[fid4] * gN[fid4])
    icT = 1 / (c * vol)
    S = d[:, :, None] * d[:, None, :] * (icT[:, None, None] + Q / 9)
    g = -d * (icT[:, None] * h.sum(1, keepdim=True) + (Q @ h[:, :, None])[:, :, 0] / 9)
    row, keep = mult[fid4], has[fid4]
    rhs = torch.zeros(L, dtype=torch.float64, device=coord.device)
    rhs.index_add_(0, row[keep], g[keep])
    if uD is not None:
        bnd = has & (torch.zeros(nF, dtype=torch.int64, device=coord.device).index_add_(
            0, fid, torch.ones_like(fid)) == 1)
        rhs[mult[bnd]] += area[bnd] * uD[bnd]
    both = keep[:, :, None] & keep[:, None, :]
    key, inv = torch.unique((row[:, :, None] * L + row[:, None, :])[both], return_inverse=True)
    values = torch.zeros(key.numel(), dtype=torch.float64, device=coord.device).index_add_(0, inv, S[both])
    iu = [0, 0, 0, 0, 1, 1, 1, 2, 2, 3], [0, 1, 2, 3, 1, 2, 3, 2, 3, 3]
    return {"values": values, "rhs": rhs, "factor": Q[:, iu[0], iu[1]] / 9, "row": key // L, "col": key % L, "L": L,
            "Q": Q, "d": d, "h": h, "icT": icT, "lrow": row, "keep": keep, "vol": vol, "P": P}


def _apply_inverse(x, w):
    """A^-1 b for b_j = (sum of w - w of the face opposite j)/3, vertex order."""
    z = x["icT"][:, None] * w.sum(1, keepdim=True) - (x["Q"] @ w[:, :, None])[:, :, 0] / 3
    return z[:, [OPP.index(j) for j in range(4)]]


def _lam_of(x, lam):
    return torch.where(x["keep"], lam[x["lrow"].clamp(min=0)], 0.0)


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _two_prod(a, b):
    def split(v):
        t = 134217729.0 * v
        hi = t - (t - v)
        return hi, v - hi
    p = a * b
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def _solve(x, b):
    """H y = b: dense Cholesky, refined with residuals in twice the precision."""
    L, row, col, val = x["L"], x["row"], x["col"], x["values"]
    H = torch.zeros((L, L), dtype=torch.float64, device=val.device)
    H[row, col] = val
    C = torch.linalg.cholesky(H)
    del H
    start = torch.searchsorted(row.contiguous(), torch.arange(L + 1, device=val.device))
    width = int((start[1:] - start[:-1]).max())
    y = torch.zeros_like(b)
    r = b
    for _ in range(6):
        y = y + torch.cholesky_solve(r[:, None], C)[:, 0]
        hi, lo = b.clone(), torch.zeros_like(b)
        for u in range(width):
            at = (start[:-1] + u).clamp(max=val.numel() - 1)
            v = torch.where(start[:-1] + u < start[1:], val[at], 0.0)
            p, e = _two_prod(v, y[col[at]])
            hi, t = _two_sum(hi, -p)
            lo = lo + (t - e)
        r = hi + lo
    return y


def exact(case, seed):
    kind = case["kind"]
    if kind == "refine":
        return _exact_refine(case, seed)
    if kind == "batch":
        s = prepare(dict(case, build=True), seed)
        out = {"values": [], "rhs": [], "factor": [], "u": []}
        for coord, tet, a, f, lam in zip(s["coord"], s["tet"], s["a"], s["f"], s["lam"]):
            x = _exact_system(coord, tet, None, a, case["c"], f, None, None)
            for k in ("values", "rhs", "factor"):
                out[k].append(x[k].reshape(-1))
            out["u"].append(_apply_inverse(x, x["h"] + x["d"] * _lam_of(x, lam)).reshape(-1))
        return {k: torch.cat(v) for k, v in out.items()}
    if kind == "gradient" and _counts(case)[3] > DENSE_MAX:
        return None
    s = prepare(case, seed)
    s = {k: v.cuda() if isinstance(v, torch.Tensor) else v for k, v in s.items()}
    x = _exact_system(s["coord"], s["tet"], s["nb"], s["a"], s["c"], s["f"], s["uD"], s["gN"])
    out = {"values": x["values"], "rhs": x["rhs"]}
    if kind in ("step", "host"):
        lam = s["lam"]
        if kind == "step":
            out["factor"] = x["factor"]
    elif x["L"] > DENSE_MAX:
        return dict(out, lam=None, u=None)
    else:
        lam = _solve(x, x["rhs"])
    u = _apply_inverse(x, x["h"] + x["d"] * _lam_of(x, lam))
    if kind == "gradient":
        return _exact_gradient(s, x, u)
    if kind == "forward":
        out["lam"] = lam
    out["u"] = u
    if case.get("pattern") or kind == "host":
        out["rowptr"] = out["colind"] = None
    return out


def _exact_gradient(s, x, u):
    e = u - s["u_obs"]
    r = x["vol"][:, None] / 20 * (e + e.sum(1, keepdim=True))  # M(T) e
    J = 0.5 * (e * r).sum()
    rf = r[:, OPP]  # face-indexed: the value at the opposite vertex
    car = x["d"] * (x["icT"][:, None] * r.sum(1, keepdim=True) - (x["Q"] @ rf[:, :, None])[:, :, 0] / 3)
    rhs = torch.zeros_like(x["rhs"]).index_add_(0, x["lrow"][x["keep"]], -car[x["keep"]])
    w = x["d"] * _lam_of(x, _solve(x, rhs))
    p = x["icT"][:, None] * r.sum(1, keepdim=True) + (x["Q"] @ rf[:, :, None])[:, :, 0]
    p = p[:, [OPP.index(j) for j in range(4)]] + _apply_inverse(x, w)
    E = x["P"][:, 1:] - x["P"][:, :1]
    cof = torch.stack([torch.linalg.cross(E[:, 1], E[:, 2]), torch.linalg.cross(E[:, 2], E[:, 0]),
                       torch.linalg.cross(E[:, 0], E[:, 1])], dim=1) / (6 * x["vol"][:, None, None])
    grad_of = lambda q: ((q[:, 1:] - q[:, :1])[:, :, None] * cof).sum(1)  # up to the sign of det E, squared below
    return {"J": J, "grad": -s["a"] * x["vol"] * (grad_of(p) * grad_of(u)).sum(1)}


def _exact_refine(case, seed):
    s = prepare(case, seed)
    coord, tet = s["coord"], s["tet"].long()
    for _ in range(case["levels"]):
        nC, nE = coord.shape[0], tet.shape[0]
        e = tet[:, EDGES].reshape(-1, 2)
        lo, hi = e.min(1).values, e.max(1).values
        eid, first = _first_rank(torch.unique(lo * nC + hi, return_inverse=True)[1])
        new = torch.arange(6 * nE, device=tet.device) == first
        before = torch.cumsum(new, 0) - new.long()
        cent = nC + torch.arange(nE, device=tet.device) + before[::6]
        mid = nC + first // 6 + 1 + before[first]
        out = torch.empty((nC + nE + int(new.sum()), 3), dtype=torch.float64, device=tet.device)
        out[:nC] = coord
        out[cent] = (((coord[tet[:, 0]] + coord[tet[:, 1]]) + coord[tet[:, 2]]) + coord[tet[:, 3]]) / 4
        out[mid[new]] = (coord[e[new, 0]] + coord[e[new, 1]]) / 2
        IJ, IK, IL, JK, JL, KL = mid.view(nE, 6).unbind(1)
        I, J, K, L = tet.unbind(1)
        kids = [(J, JK, IJ, JL), (K, IK, JK, KL), (L, KL, JL, IL), (IJ, IK, IL, cent), (JK, IJ, JL, cent),
                (IK, JK, KL, cent), (KL, JL, IL, cent), (IJ, JK, IK, cent), (IK, KL, IL, cent), (IJ, IL, JL, cent),
                (KL, JK, JL, cent)]
        rest = torch.stack([torch.stack(k, dim=1) for k in kids], dim=1).reshape(-1, 4)
        coord, tet = out, torch.cat([torch.stack([I, IJ, IK, IL], dim=1), rest])
    return {"coord": coord, "tet": None, **({"neumann": None} if s["nb"] is not None else {})}
