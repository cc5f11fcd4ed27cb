"""The work that a user of this library has it do, as cases with sizes.

A case is a dict of plain values; its "kind" says which public entry points run:

  eval    one structure: Model.set_design, solve, gradient, result
  batch   many designs of one shell at once: Batch.solve, gradient, results stacked
  train   a batch inside torch.autograd: BatchSSOFunction forward and backward of a mean loss
  serve   a stream of requests of uneven size through the continuous-batching Server
  bridge  a chain of beams solved directly (precond "chain") and its sensitivities
  quads, beams   element matrices alone
  spmv    the block-sparse product y = K x with x^T y

The structures are the ones of the benchmark and tests: beam grid-shells (square node grid,
one diagonal per cell, pinned boundary), quad shells over a bump (corners pinned under
self-weight, or clamped edges under pressure) and multi-span arch bridges.  Every number of a
structure that a designer varies (heights, thicknesses, densities) comes from the seed.

`exact` forms the same element matrices with torch in 64 bits, factors K as a block-tridiagonal
matrix (one block per grid row) with one refinement, and differentiates the element energies
with autograd.
"""
import math

import numpy as np
import torch

DEV = "cuda"
PINNED = (1, 1, 1, 0, 0, 0)


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # one evaluation inside a designer's interactive loop: heights up from the host, u, C and
        # dC/dz back to it (10 x 10 nodes, 600 DOF); latency is everything
        {"name": "gridshell10", "kind": "eval", "mesh": "gridshell", "size": 10,
         "precision": "f32x2", "precond": "block_jacobi", "rtol": 1e-10, "objective": "C",
         "simp": False, "host": True},
        # FP64 CG of a mid-size grid-shell with a displacement objective J = C + g.u, so that a
        # second (adjoint) solve runs
        {"name": "gridshell41_fp64_adjoint", "kind": "eval", "mesh": "gridshell", "size": 41,
         "precision": "fp64", "precond": "block_jacobi", "rtol": 1e-10, "objective": "C+gu",
         "simp": False, "host": False},
        # one step of a topology optimisation: a small shell with element densities, the
        # stronger preconditioner
        {"name": "shell33_simp_two_level", "kind": "eval", "mesh": "shell", "size": 33,
         "precision": "fp32_ir", "precond": "two_level", "rtol": 1e-8, "objective": "C",
         "simp": True, "host": False},
        # one design of the benchmark's shell with the library's default options
        {"name": "shell64", "kind": "eval", "mesh": "shell", "size": 64,
         "precision": "fp32_ir", "precond": "block_jacobi", "rtol": 1e-8, "objective": "C",
         "simp": False, "host": False},
        # a sweep over designs of that shell at the benchmark's tolerance
        {"name": "shell64_x48", "kind": "batch", "size": 64, "designs": 48,
         "precond": "block_jacobi", "rtol": 1e-6},
        # a larger sweep with the two-level preconditioner
        {"name": "shell64_x128_two_level", "kind": "batch", "size": 64, "designs": 128,
         "precond": "two_level", "rtol": 1e-6},
        # one training step's physics: 24 shells of 48 x 48 elements, loss = mean(C + 0.1 V),
        # gradients to heights and thicknesses through autograd
        {"name": "train48_x24", "kind": "train", "size": 48, "designs": 24,
         "precond": "block_jacobi", "rtol": 1e-6},
        # 64 queued grid-shell requests of 8 x 8 to 100 x 100 nodes (384 to 60,000 DOF) from host
        # memory and back to it
        {"name": "serve64", "kind": "serve", "requests": 64, "side_min": 8, "side_max": 100,
         "precond": "block_jacobi", "rtol": 1e-6, "lanes": 2},
        # one large shell, clamped edges under pressure, Jacobi (396,294 DOF; K alone 85 MB)
        {"name": "shell256_clamped", "kind": "eval", "mesh": "shell_clamped", "size": 256,
         "precision": "fp32_ir", "precond": "jacobi", "rtol": 1e-8, "objective": "C",
         "simp": False, "host": False},
        # sensitivities of a 100-span bridge, 900,006 DOF, direct solve
        {"name": "bridge1500", "kind": "bridge", "el_per_span": 1500},
        # element matrices of a 512 x 512 mesh
        {"name": "quads262144", "kind": "quads", "count": 262144},
        # one product with the assembled K of a 256 x 256 shell (66,049 nodes, 170 MB of K)
        {"name": "spmv66049", "kind": "spmv", "side": 257},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "batch", "batch", "train", "serve", "bridge",
                       "quads", "beams", "spmv"])
    if kind == "eval":
        mesh = rng.choice(["gridshell", "shell", "shell_clamped"])
        precision = rng.choice(["f32x2", "fp64", "fp32_ir", "fp32_ir"])
        if precision == "f32x2":  # small systems only
            size = _log_int(rng, 8, 20) if mesh == "gridshell" else _log_int(rng, 5, 12)
            rtol = 1e-10
        elif precision == "fp64":
            size = _log_int(rng, 8, 60) if mesh == "gridshell" else _log_int(rng, 5, 24)
            rtol = 1e-10
        else:
            size = (_log_int(rng, 8, 100) if mesh == "gridshell" else
                    _log_int(rng, 8, 72) if mesh == "shell" else _log_int(rng, 16, 256))
            rtol = rng.choice([1e-6, 1e-8])
        precond = rng.choice(["block_jacobi", "jacobi", "two_level"])
        if precision == "fp64" and precond == "two_level":
            precond = "block_jacobi"
        return {"kind": "eval", "mesh": mesh, "size": size, "precision": precision,
                "precond": precond, "rtol": rtol,
                "objective": rng.choice(["C", "C", "C+gu"]),
                "simp": mesh != "gridshell" and rng.random() < 0.3, "host": rng.random() < 0.5}
    if kind == "batch":
        size, precond = rng.randint(16, 64), rng.choice(["block_jacobi", "two_level"])
        most = 48 if precond == "block_jacobi" else 128
        return {"kind": "batch", "size": size, "designs": _log_int(rng, 2, most),
                "precond": precond, "rtol": rng.choice([1e-6, 1e-8]) if size < 48 else 1e-6}
    if kind == "train":
        return {"kind": "train", "size": rng.randint(16, 48), "designs": _log_int(rng, 2, 24),
                "precond": rng.choice(["block_jacobi", "two_level"]), "rtol": 1e-6}
    if kind == "serve":
        hi = rng.randint(24, 100)
        return {"kind": "serve", "requests": _log_int(rng, 4, 64), "side_min": 8, "side_max": hi,
                "precond": rng.choice(["block_jacobi", "two_level"]), "rtol": 1e-6,
                "lanes": rng.choice([1, 2])}
    if kind == "bridge":
        return {"kind": "bridge", "el_per_span": _log_int(rng, 2, 1500)}
    if kind == "spmv":
        return {"kind": "spmv", "side": _log_int(rng, 20, 257)}
    return {"kind": kind, "count": _log_int(rng, 500, 262144)}


# ---------------------------------------------------------------------------
# structures (plain numpy)

def _empty(n):
    return {"xyz": np.zeros((n, 3)), "beam_conn": np.zeros((0, 2), np.int32),
            "beam_props": np.zeros((0, 6)), "quad_conn": np.zeros((0, 4), np.int32),
            "quad_props": np.zeros((0, 5)), "fixed": np.zeros((n, 6), np.uint8),
            "nodal_load": np.zeros((n, 6)), "pressure": 0.0, "gamma": 0.0}


def _grid(side, span):
    s = np.linspace(0.0, span, side)
    xx, yy = np.meshgrid(s, s, indexing="xy")
    return xx.ravel(), yy.ravel()


def _gridshell_z(side, seed):
    """A sum of four sinusoids of at most 0.5 m each over a 10 m plan."""
    rng = np.random.default_rng(seed)
    x, y = _grid(side, 10.0)
    a, phi = rng.uniform(0.0, 0.5, 4), rng.uniform(0.0, 2 * math.pi, 4)
    m, n = rng.integers(1, 4, 4), rng.integers(1, 4, 4)
    return sum(a[k] * np.sin(2 * math.pi * (m[k] * x + n[k] * y) / 10.0 + phi[k])
               for k in range(4))


def _gridshell(side, seed):
    """Steel tubes along every grid edge and one diagonal per cell, 1 kN at every free node."""
    x, y = _grid(side, 10.0)
    m = _empty(side * side)
    m["xyz"] = np.stack([x, y, _gridshell_z(side, seed)], axis=1)
    nid = np.arange(side * side, dtype=np.int32).reshape(side, side)
    pairs = [(nid[:, :-1], nid[:, 1:]), (nid[:-1, :], nid[1:, :]), (nid[:-1, :-1], nid[1:, 1:])]
    m["beam_conn"] = np.concatenate(
        [np.stack([a.ravel(), b.ravel()], 1) for a, b in pairs]).astype(np.int32)
    area = math.pi * (0.05 ** 2 - 0.045 ** 2)
    inertia = math.pi / 4 * (0.05 ** 4 - 0.045 ** 4)
    E = 210e9
    m["beam_props"] = np.tile([E, E / 2.6, inertia, inertia, 2 * inertia, area],
                              (m["beam_conn"].shape[0], 1))
    edge = np.ones((side, side), bool)
    edge[1:-1, 1:-1] = False
    m["fixed"][edge.ravel()] = PINNED
    m["nodal_load"][~edge.ravel(), 2] = -1000.0
    return m


def _shell_design(n_el, seed):
    """Heights of a smooth bump of 5 m over a 20 m plan, thicknesses in [0.05, 0.2] m."""
    rng = np.random.default_rng(seed)
    x, y = _grid(n_el + 1, 20.0)
    b, phi = rng.uniform(0.0, 1.0, 2), rng.uniform(0.0, 2 * math.pi, 2)
    m, n = rng.integers(1, 4, 2), rng.integers(1, 4, 2)
    s = np.sin(math.pi * x / 20) * np.sin(math.pi * y / 20) * (
        1 + sum(0.2 * b[k] * np.sin(2 * math.pi * (m[k] * x + n[k] * y) / 20 + phi[k])
                for k in range(2)))
    return 5.0 * s / s.max(), rng.uniform(0.05, 0.2, n_el * n_el)


def _shell(n_el, z, t, clamped=False):
    side = n_el + 1
    x, y = _grid(side, 20.0)
    m = _empty(side * side)
    m["xyz"] = np.stack([x, y, z], axis=1)
    nid = np.arange(side * side, dtype=np.int32).reshape(side, side)
    m["quad_conn"] = np.stack([nid[:-1, :-1].ravel(), nid[:-1, 1:].ravel(), nid[1:, 1:].ravel(),
                               nid[1:, :-1].ravel()], 1).astype(np.int32)
    m["quad_props"] = np.tile([0.1, 30e9, 0.2, 1.0, 1.0], (n_el * n_el, 1))
    m["quad_props"][:, 0] = t
    if clamped:
        edge = np.ones((side, side), bool)
        edge[1:-1, 1:-1] = False
        m["fixed"][edge.ravel()] = 1
        m["pressure"] = 5e3
    else:
        m["fixed"][[nid[0, 0], nid[0, -1], nid[-1, 0], nid[-1, -1]]] = PINNED
        m["gamma"] = 25e3
    return m


def _bridge(el_per_span, seed, spans=100):
    """100 parabolic arches of 30 m on pinned piers, each of a rise of its own around 10 m, with
    their self-weight as nodal loads."""
    rise = np.random.default_rng(seed).uniform(8.0, 12.0, spans)
    n = spans * el_per_span + 1
    m = _empty(n)
    xi = (np.arange(n) % el_per_span) / el_per_span
    span_of = np.minimum(np.arange(n) // el_per_span, spans - 1)
    m["xyz"][:, 0] = np.arange(n) * (30.0 / el_per_span)
    m["xyz"][:, 2] = 4.0 * rise[span_of] * xi * (1 - xi)
    m["beam_conn"] = np.stack([np.arange(n - 1), np.arange(1, n)], 1).astype(np.int32)
    m["beam_props"] = np.tile([2e11, 2e11 / 2.6, 6.6e-5, 3.3e-6, 6.93e-5, 4.3e-3], (n - 1, 1))
    m["fixed"][::el_per_span] = (1, 1, 1, 1, 0, 1)
    length = np.linalg.norm(np.diff(m["xyz"], axis=0), axis=1)
    m["nodal_load"][:-1, 2] -= 0.5 * 7.85e4 * 4.3e-3 * length
    m["nodal_load"][1:, 2] -= 0.5 * 7.85e4 * 4.3e-3 * length
    return m


def _eval_mesh(case, seed):
    if case["mesh"] == "gridshell":
        return _gridshell(case["size"], seed)
    z, t = _shell_design(case["size"], seed)
    return _shell(case["size"], z, t, case["mesh"] == "shell_clamped")


def _eval_extra(case, seed, n_nodes, n_quads):
    """Objective vector g (J = C + g.u; a few nodes' displacements watched) and densities."""
    rng = np.random.default_rng(seed + 77)
    g = rho = None
    if case["objective"] == "C+gu":
        g = np.zeros((n_nodes, 6))
        g[rng.integers(0, n_nodes, 8), 2] = rng.uniform(500.0, 1500.0, 8)
    if case["simp"]:
        rho = rng.uniform(0.3, 1.0, n_quads)
    return g, rho


def _train_design(case, seed):
    rng = np.random.default_rng(seed)
    z0, _ = _shell_design(case["size"], seed)
    z = np.stack([z0 + 0.25 * np.tanh(0.5 * rng.standard_normal(z0.shape))
                  for _ in range(case["designs"])])
    return z, np.full((case["designs"], case["size"] ** 2), 0.1)


def _serve_meshes(case, seed):
    """Sides spread over the range, in a seeded order: the stream's work does not depend on luck."""
    rng = np.random.default_rng(seed)
    sides = np.linspace(case["side_min"], case["side_max"], case["requests"]).round().astype(int)
    return [_gridshell(int(s), int(rng.integers(1 << 30))) for s in rng.permutation(sides)]


def _loose_quads(count, seed):
    """Elements of a curved mesh row: corners on a jittered, warped strip."""
    rng = np.random.default_rng(seed)
    cols = max(2, int(math.sqrt(count)))
    rows = -(-count // cols)
    x, y = np.meshgrid(np.arange(cols + 1) * 0.3, np.arange(rows + 1) * 0.3, indexing="xy")
    xyz = np.stack([x.ravel(), y.ravel(), np.sin(x.ravel() / 3) + np.cos(y.ravel() / 4)], 1)
    xyz += rng.uniform(-0.03, 0.03, xyz.shape)
    nid = np.arange((cols + 1) * (rows + 1)).reshape(rows + 1, cols + 1)
    conn = np.stack([nid[:-1, :-1].ravel(), nid[:-1, 1:].ravel(), nid[1:, 1:].ravel(),
                     nid[1:, :-1].ravel()], 1)[:count]
    props = np.tile([0.1, 30e9, 0.2, 1.0, 1.0], (count, 1))
    props[:, 0] = rng.uniform(0.05, 0.2, count)
    return xyz, conn.astype(np.int32), props


def _loose_beams(count, seed):
    rng = np.random.default_rng(seed)
    xyz = rng.uniform(0.0, 10.0, (count // 3 + 2, 3))
    i = rng.integers(0, len(xyz), count)
    j = (i + rng.integers(1, len(xyz), count)) % len(xyz)
    props = np.tile([210e9, 81e9, 1.7e-6, 1.7e-6, 3.4e-6, 1.5e-3], (count, 1))
    props[:, 2:6] *= rng.uniform(0.5, 2.0, (count, 4))
    return xyz, np.stack([i, j], 1).astype(np.int32), props


def _spmv_inputs(side, seed):
    """A 9-point block pattern on a side x side node grid with random blocks."""
    n = side * side
    i, j = np.divmod(np.arange(n), side)
    cols = []
    for di in (-1, 0, 1):
        for dj in (-1, 0, 1):
            ok = (i + di >= 0) & (i + di < side) & (j + dj >= 0) & (j + dj < side)
            cols.append(np.where(ok, (i + di) * side + j + dj, -1))
    cols = np.stack(cols, 1)
    row_ptr = np.concatenate([[0], np.cumsum((cols >= 0).sum(1))]).astype(np.int32)
    col = cols[cols >= 0].astype(np.int32)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    K = torch.randn(len(col), 6, 6, dtype=torch.float64, device=DEV, generator=gen)
    x = torch.randn(6 * n, dtype=torch.float64, device=DEV, generator=gen)
    return torch.tensor(row_ptr, device=DEV), torch.tensor(col, device=DEV), K, x


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass

def _dev(a, dtype=torch.float64):
    return torch.tensor(a, dtype=dtype, device=DEV)


def prepare(case, seed):
    import paper_2407_20026_gb300 as sso

    kind = case["kind"]
    s = {"case": case, "sso": sso}
    if kind == "eval":
        m = _eval_mesh(case, seed)
        s["model"] = sso.Model(m)
        put = (lambda a: a) if case["host"] else _dev
        s["z"] = put(np.ascontiguousarray(m["xyz"][:, 2]))
        s["t"] = put(np.ascontiguousarray(m["quad_props"][:, 0])) if len(m["quad_conn"]) else None
        g, rho = _eval_extra(case, seed, len(m["xyz"]), len(m["quad_conn"]))
        s["g"] = None if g is None else put(g.ravel())
        s["rho"] = None if rho is None else put(rho)
        s["opts"] = sso.options(precision=case["precision"], precond=case["precond"],
                                rtol=case["rtol"])
    elif kind == "batch":
        designs = [_shell_design(case["size"], seed * 1000 + k) for k in range(case["designs"])]
        s["batch"] = sso.Batch([sso.Model(_shell(case["size"], z, t)) for z, t in designs])
        s["z"] = [_dev(z) for z, _ in designs]
        s["t"] = [_dev(t) for _, t in designs]
        s["opts"] = sso.options(precond=case["precond"], rtol=case["rtol"])
    elif kind == "train":
        z, t = _train_design(case, seed)
        base = _shell(case["size"], z[0], t[0])
        s["batch"] = sso.Batch([sso.Model(base) for _ in range(case["designs"])])
        s["z"], s["t"] = _dev(z), _dev(t)
        s["opts"] = sso.options(precond=case["precond"], rtol=case["rtol"])
    elif kind == "serve":
        from paper_2407_20026_gb300.serve import Server
        s["meshes"] = _serve_meshes(case, seed)
        s["server"] = Server(sso.options(precond=case["precond"], rtol=case["rtol"]),
                             hbm_budget=6 << 30, max_systems=256, lanes=case["lanes"])
    elif kind == "bridge":
        m = _bridge(case["el_per_span"], seed)
        s["model"] = sso.Model(m)
        s["z"] = _dev(np.ascontiguousarray(m["xyz"][:, 2]))
        s["opts"] = sso.options(precision="fp64", precond="chain", rtol=1e-10, max_sweeps=3)
    elif kind in ("quads", "beams"):
        xyz, conn, props = (_loose_quads if kind == "quads" else _loose_beams)(case["count"], seed)
        s["args"] = (_dev(xyz), _dev(conn, torch.int32), _dev(props))
    elif kind == "spmv":
        s["args"] = _spmv_inputs(case["side"], seed)
    return s


def run(s):
    sso, kind = s["sso"], s["case"]["kind"]
    if kind == "eval":
        m, dev = s["model"], None if s["case"]["host"] else DEV
        m.set_design(s["z"], s["t"])
        if s["rho"] is not None:
            m.set_topology(s["rho"], 3.0)
        m.solve(s["opts"])
        m.gradient(1.0, s["g"])
        r = m.result(device=dev)
        out = {"u": r["u"], "C": r["C"], "dz": r["dz"]}
        if s["t"] is not None:
            out["dt"] = r["dt"]
        if s["rho"] is not None:
            out["drho"] = m.topology_gradient(device=dev)
        return out
    if kind == "batch":
        b = s["batch"]
        for m, z, t in zip(b.models, s["z"], s["t"]):
            m.set_design(z, t)
        b.solve(s["opts"])
        b.gradient()
        r = [m.result(device=DEV) for m in b.models]
        return {"u": torch.stack([x["u"] for x in r]), "C": np.array([x["C"] for x in r]),
                "dz": torch.stack([x["dz"] for x in r]), "dt": torch.stack([x["dt"] for x in r])}
    if kind == "train":
        from paper_2407_20026_gb300.autograd import BatchSSOFunction
        z, t = s["z"].detach().requires_grad_(True), s["t"].detach().requires_grad_(True)
        u, C, V = BatchSSOFunction.apply(s["batch"], z, t, s["opts"])
        (C + 0.1 * V).mean().backward()
        return {"u": u.detach(), "C": C.detach(), "V": V.detach(), "dz": z.grad, "dt": t.grad}
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(m) for m in s["meshes"]]
        while True:
            resident, waiting = srv.step()
            if resident == 0 and waiting == 0:
                break
        srv.completed()
        r = [srv.poll(t) for t in tickets]
        return {"u": np.concatenate([x["u"] for x in r]), "C": np.array([x["C"] for x in r]),
                "dz": np.concatenate([x["dz"] for x in r])}
    if kind == "bridge":
        m = s["model"]
        m.set_design(s["z"])
        m.solve(s["opts"], raise_on_error=False)
        m.gradient()
        r = m.result(device=DEV)
        return {"u": r["u"], "C": r["C"], "dz": r["dz"]}
    if kind == "quads":
        return sso.model.quad_stiffness(*s["args"])
    if kind == "beams":
        return sso.model.beam_stiffness(*s["args"])
    return sso.model.bsr_spmv(*s["args"])


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _counts(mesh, size):
    """(nodes, K blocks, elements, bytes of the mesh's designable inputs)."""
    if mesh == "gridshell":
        n, e = size * size, 2 * size * (size - 1) + (size - 1) ** 2
        return n, n + 2 * e, e, 8 * n
    side = size + 1
    n = side * side
    return n, n + 4 * size * side + 4 * size * size, size * size, 8 * (n + size * size)


def _iterations(mesh, size, precond, rtol):
    """CG iterations that a structure of this kind takes, roughly: they grow with the side."""
    per = {"gridshell": 25.0, "shell": 190.0, "shell_clamped": 30.0}[mesh]
    per *= {"jacobi": 1.3, "block_jacobi": 1.0, "two_level": 0.2}[precond]
    return per * size * -math.log10(rtol) / 6.0


def _solve_work(mesh, size, precond, rtol, solves=1, outputs=0):
    n, blocks, elements, inputs = _counts(mesh, size)
    return {"bytes": inputs + 8 * (7 * n + 1 + outputs),
            "flops": solves * 72.0 * blocks * _iterations(mesh, size, precond, rtol)
            + elements * (6e3 if mesh != "gridshell" else 1e3)}


def work(case):
    kind = case["kind"]
    if kind == "eval":
        extra = case["size"] ** 2 * (case["mesh"] != "gridshell") * (1 + 2 * case["simp"])
        return _solve_work(case["mesh"], case["size"], case["precond"], case["rtol"],
                           2 if case["objective"] == "C+gu" else 1, extra)
    if kind in ("batch", "train"):
        w = _solve_work("shell", case["size"], case["precond"], case["rtol"], 1,
                        case["size"] ** 2)
        return {k: case["designs"] * v for k, v in w.items()}
    if kind == "serve":
        sides = np.linspace(case["side_min"], case["side_max"], case["requests"]).round()
        ws = [_solve_work("gridshell", int(s), case["precond"], case["rtol"]) for s in sides]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "bridge":
        n = 100 * case["el_per_span"] + 1
        return {"bytes": 8 * (n + 7 * n), "flops": 2000.0 * n}
    if kind == "quads":
        return {"bytes": case["count"] * (12 * 8 + 16 + 40 + 576 * 8), "flops": case["count"] * 6e3}
    if kind == "beams":
        return {"bytes": case["count"] * (6 * 8 + 8 + 48 + 144 * 8), "flops": case["count"] * 1e3}
    n = case["side"] ** 2
    blocks = (3 * case["side"] - 2) ** 2
    return {"bytes": blocks * 292 + n * (2 * 48 + 4), "flops": 72.0 * blocks}


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch

def _quad_matrices(X, t, E, nu):
    """X [e, 4, 3], t, E [e] -> k_e [e, 24, 24] (global axes) and the facet's nodal area shares
    [e, 4].  Flat facet on the mean plane; membrane, bending, assumed transverse shear tied at
    the edge mid-points, drilling penalty; 2 x 2 Gauss; rigid links from the warped nodes."""
    c = X.mean(1)
    n = torch.linalg.cross(X[:, 2] - X[:, 0], X[:, 3] - X[:, 1])
    n = n / n.norm(dim=1, keepdim=True)
    a = (X[:, 1] - X[:, 0]) + (X[:, 2] - X[:, 3])
    a = a - (a * n).sum(1, keepdim=True) * n
    e1 = a / a.norm(dim=1, keepdim=True)
    R = torch.stack([e1, torch.linalg.cross(n, e1), n], 1)
    loc = torch.einsum("erk,eak->ear", R, X - c[:, None])
    x, y, h = loc[..., 0], loc[..., 1], loc[..., 2]
    xin, etan = (torch.tensor(v, dtype=X.dtype, device=X.device)
                 for v in ([-1.0, 1, 1, -1], [-1.0, -1, 1, 1]))
    ne = X.shape[0]

    def point(xi, eta):
        N = 0.25 * (1 + xin * xi) * (1 + etan * eta)
        dxi, deta = 0.25 * xin * (1 + etan * eta), 0.25 * etan * (1 + xin * xi)
        return N, dxi, deta, x @ dxi, y @ dxi, x @ deta, y @ deta

    def row(cols):
        B = [None] * 24
        zero = torch.zeros(ne, dtype=X.dtype, device=X.device)
        for (node, dof), v in cols.items():
            B[6 * node + dof] = v
        return torch.stack([zero if v is None else v for v in B], 1)

    def tying(xi, eta, along_xi):
        N, dxi, deta, xxi, yxi, xeta, yeta = point(xi, eta)
        d, dx, dy = (dxi, xxi, yxi) if along_xi else (deta, xeta, yeta)
        cols = {}
        for i in range(4):
            cols[i, 2] = d[i].expand(ne)
            cols[i, 3] = -N[i] * dy
            cols[i, 4] = N[i] * dx
        return row(cols)

    tB, tD, tA, tC = tying(0, -1, True), tying(0, 1, True), tying(-1, 0, False), tying(1, 0, False)
    G = E / (2 * (1 + nu))
    cm, cb = E / (1 - nu * nu) * t, E / (12 * (1 - nu * nu)) * t ** 3
    D = torch.tensor([[1, nu, 0], [nu, 1, 0], [0, 0, (1 - nu) / 2]], dtype=X.dtype, device=X.device)
    k = torch.zeros(ne, 24, 24, dtype=X.dtype, device=X.device)
    area = torch.zeros(ne, 4, dtype=X.dtype, device=X.device)
    gp = 1 / math.sqrt(3.0)
    for eta in (-gp, gp):
        for xi in (-gp, gp):
            N, dxi, deta, xxi, yxi, xeta, yeta = point(xi, eta)
            det = xxi * yeta - yxi * xeta
            Nx = (yeta[:, None] * dxi - yxi[:, None] * deta) / det[:, None]
            Ny = (xxi[:, None] * deta - xeta[:, None] * dxi) / det[:, None]
            mx, my, mxy, bx, by, bxy, dr = ({} for _ in range(7))
            for i in range(4):
                mx[i, 0], my[i, 1], mxy[i, 0], mxy[i, 1] = Nx[:, i], Ny[:, i], Ny[:, i], Nx[:, i]
                bx[i, 4], by[i, 3], bxy[i, 4], bxy[i, 3] = Nx[:, i], -Ny[:, i], Ny[:, i], -Nx[:, i]
                dr[i, 0], dr[i, 1], dr[i, 5] = 0.5 * Ny[:, i], -0.5 * Nx[:, i], N[i].expand(ne)
            gx = 0.5 * (1 - eta) * tB + 0.5 * (1 + eta) * tD
            ge = 0.5 * (1 - xi) * tA + 0.5 * (1 + xi) * tC
            s1 = (yeta[:, None] * gx - yxi[:, None] * ge) / det[:, None]
            s2 = (xxi[:, None] * ge - xeta[:, None] * gx) / det[:, None]
            for rows, W in (((mx, my, mxy), cm[:, None, None] * D),
                            ((bx, by, bxy), cb[:, None, None] * D)):
                B = torch.stack([row(r) for r in rows], 1)
                k = k + det[:, None, None] * (B.transpose(1, 2) @ W @ B)
            B = torch.stack([s1, s2], 1)
            k = k + (det * 5 / 6 * G * t)[:, None, None] * (B.transpose(1, 2) @ B)
            B = row(dr)[:, None]
            k = k + (det * 0.01 * G * t)[:, None, None] * (B.transpose(1, 2) @ B)
            area = area + det[:, None] * N
    T = torch.zeros(ne, 24, 24, dtype=X.dtype, device=X.device)
    for i in range(4):
        blk = torch.zeros(ne, 6, 6, dtype=X.dtype, device=X.device)
        blk[:, :3, :3] = R
        blk[:, 3:, 3:] = R
        blk[:, 0, 3:] = -h[:, i, None] * R[:, 1]
        blk[:, 1, 3:] = h[:, i, None] * R[:, 0]
        T[:, 6 * i:6 * i + 6, 6 * i:6 * i + 6] = blk
    return T.transpose(1, 2) @ k @ T, area


def _beam_matrices(X, p):
    """X [e, 2, 3], p [e, 6] = E, G, Iy, Iz, J, A -> k_e [e, 12, 12] in global axes."""
    d = X[:, 1] - X[:, 0]
    L = d.norm(dim=1)
    ex = d / L[:, None]
    upright = ex[:, 2].abs() > 1 - 1e-8
    hn = torch.where(upright, torch.ones_like(L), ex[:, 0] ** 2 + ex[:, 1] ** 2).sqrt()
    ey = torch.where(upright[:, None], torch.tensor([0.0, 1.0, 0.0], dtype=X.dtype, device=X.device),
                     torch.stack([-ex[:, 1] / hn, ex[:, 0] / hn, torch.zeros_like(L)], 1))
    R = torch.stack([ex, ey, torch.linalg.cross(ex, ey)], 1)
    E, G, Iy, Iz, J, A = p.unbind(1)
    k = torch.zeros(len(L), 12, 12, dtype=X.dtype, device=X.device)

    def put(i, j, v):
        k[:, i, j] = v
        if i != j:
            k[:, j, i] = v

    for a, v in ((0, E * A / L), (3, G * J / L)):
        put(a, a, v), put(a + 6, a + 6, v), put(a, a + 6, -v)
    for v, r, sg, EI in ((1, 5, 1.0, E * Iz), (2, 4, -1.0, E * Iy)):
        put(v, v, 12 * EI / L ** 3), put(v + 6, v + 6, 12 * EI / L ** 3)
        put(v, v + 6, -12 * EI / L ** 3)
        put(r, r, 4 * EI / L), put(r + 6, r + 6, 4 * EI / L), put(r, r + 6, 2 * EI / L)
        b = sg * 6 * EI / L ** 2
        put(v, r, b), put(v, r + 6, b), put(v + 6, r, -b), put(v + 6, r + 6, -b)
    T = torch.zeros_like(k)
    for i in range(4):
        T[:, 3 * i:3 * i + 3, 3 * i:3 * i + 3] = R
    return T.transpose(1, 2) @ k @ T


class _Exact:
    """Structures of one topology (designs in the leading dimension d): K as a block-tridiagonal
    matrix of `per` nodes a block, factored once."""

    def __init__(self, m, z, per, t=None, rho=None):
        self.m, self.per = m, per
        self.z = z.clone().requires_grad_(True)
        self.nd, self.n = z.shape
        self.t = self.rho = None
        if t is not None:
            self.t = t.clone().requires_grad_(True)
            self.rho = (torch.ones_like(t) if rho is None else rho).clone().requires_grad_(True)
        self.xy = _dev(m["xyz"][:, :2])
        self.bc = _dev(m["beam_conn"], torch.int64)
        self.qc = _dev(m["quad_conn"], torch.int64)
        self.free = _dev(1.0 - (m["fixed"].ravel() != 0))
        self.nodal = _dev(m["nodal_load"].ravel())
        with torch.no_grad():
            parts = [self.elements(k) for k in range(self.nd)]
            self.ke = [torch.stack([q[i] for q in parts]) if parts[0][i] is not None else None
                       for i in (0, 1)]
            self.f = torch.stack([q[2] for q in parts]) * self.free
            self.factor()

    def elements(self, k):
        """(k_e of the beams, of the quads, load vector) of design k."""
        m = self.m
        X = torch.cat([self.xy, self.z[k][:, None]], 1)
        f, kb, kq = self.nodal, None, None
        if len(self.bc):
            kb = _beam_matrices(X[self.bc], _dev(m["beam_props"]))
        if len(self.qc):
            E0, nu = _dev(m["quad_props"][:, 1]), float(m["quad_props"][0, 2])
            kq, area = _quad_matrices(X[self.qc], self.t[k], self.rho[k] ** 3 * E0, nu)
            share = -(m["pressure"] + m["gamma"] * self.t[k])[:, None] * area
            f = f.index_add(0, (6 * self.qc + 2).ravel(), share.ravel())
        return kb, kq, f

    def sets(self):
        for conn, ke in zip((self.bc, self.qc), self.ke):
            if ke is not None:
                yield (6 * conn[:, :, None] + torch.arange(6, device=DEV)).flatten(1), ke

    def factor(self):
        w = 6 * self.per
        rows = -(-6 * self.n // w)
        D = torch.zeros(self.nd, rows, w, w, dtype=torch.float64, device=DEV)
        U = torch.zeros(self.nd, rows, w, w, dtype=torch.float64, device=DEV)
        for dof, ke in self.sets():
            i, j = dof[:, :, None].expand_as(ke[0]), dof[:, None, :].expand_as(ke[0])
            v = ke * (self.free[i] * self.free[j])
            for to, shift in ((D, 0), (U, 1)):
                pick = (j // w - i // w) == shift
                at = ((i // w) * w + i % w) * w + j % w
                for k in range(self.nd):
                    to[k].view(-1).index_add_(0, at[pick], v[k][pick])
        held = torch.cat([1 - self.free, torch.ones(rows * w - 6 * self.n, dtype=torch.float64,
                                                    device=DEV)])
        torch.diagonal(D, dim1=2, dim2=3).add_(held.view(rows, w))
        self.L, self.W = [], []
        for r in range(rows):
            S = D[:, r]
            if r:
                S = S - self.W[-1].transpose(1, 2) @ self.W[-1]
            # one matrix at a time: each is a few hundred wide
            self.L.append(torch.stack([torch.linalg.cholesky(S[k]) for k in range(self.nd)]))
            if r + 1 < rows:
                self.W.append(torch.linalg.solve_triangular(self.L[-1], U[:, r], upper=False))
        self.pad = rows * w - 6 * self.n

    def direct(self, b):
        b = torch.nn.functional.pad(b, (0, self.pad)).view(self.nd, len(self.L), -1, 1)
        y, x = [], [None] * len(self.L)
        for r, L in enumerate(self.L):
            v = b[:, r] if r == 0 else b[:, r] - self.W[r - 1].transpose(1, 2) @ y[-1]
            y.append(torch.linalg.solve_triangular(L, v, upper=False))
        for r in reversed(range(len(self.L))):
            v = y[r] if r + 1 == len(self.L) else y[r] - self.W[r] @ x[r + 1]
            x[r] = torch.linalg.solve_triangular(self.L[r].transpose(1, 2), v, upper=True)
        return torch.stack(x, 1).view(self.nd, -1)[:, :6 * self.n] * self.free

    def product(self, u):
        y = torch.zeros_like(u)
        for dof, ke in self.sets():
            v = (ke @ u[:, dof].unsqueeze(-1)).flatten(1)
            y.index_add_(1, dof.ravel(), v)
        return y * self.free

    def solve(self, b):
        with torch.no_grad():
            x = self.direct(b)
            return x + self.direct(b - self.product(x))

    def gradients(self, u, lam, weight):
        """d/d(z, t, rho) of lam.(f - K u) + weight f.u, per design."""
        for k in range(self.nd):
            kb, kq, f = self.elements(k)
            J = ((lam[k] + weight * u[k]) * f * self.free).sum()
            for conn, ke in ((self.bc, kb), (self.qc, kq)):
                if ke is not None:
                    dof = (6 * conn[:, :, None] + torch.arange(6, device=DEV)).flatten(1)
                    J = J - torch.einsum("ei,eij,ej->", lam[k][dof], ke, u[k][dof])
            J.backward()
        return self.z.grad, None if self.t is None else self.t.grad, \
            None if self.rho is None else self.rho.grad


def exact(case, seed):
    kind = case["kind"]
    if kind == "eval":
        m = _eval_mesh(case, seed)
        g, rho = _eval_extra(case, seed, len(m["xyz"]), len(m["quad_conn"]))
        side = case["size"] + (case["mesh"] != "gridshell")
        t = _dev(m["quad_props"][None, :, 0]) if len(m["quad_conn"]) else None
        X = _Exact(m, _dev(m["xyz"][None, :, 2]), side, t, None if rho is None else _dev(rho[None]))
        u = X.solve(X.f)
        lam = u if g is None else X.solve(X.f + _dev(g.ravel()) * X.free)
        dz, dt, drho = X.gradients(u, lam, 1.0)
        out = {"u": u[0], "C": (X.f * u).sum(), "dz": dz[0]}
        if t is not None:
            out["dt"] = dt[0]
        if rho is not None:
            out["drho"] = drho[0]
        return out
    if kind in ("batch", "train"):
        if kind == "batch":
            z, t = (np.stack(v) for v in zip(*[_shell_design(case["size"], seed * 1000 + k)
                                               for k in range(case["designs"])]))
        else:
            z, t = _train_design(case, seed)
        parts = []
        for k in range(0, len(z), 16):  # a few at a time: the factors are dense blocks
            m = _shell(case["size"], z[k], t[k])
            X = _Exact(m, _dev(z[k:k + 16]), case["size"] + 1, _dev(t[k:k + 16]))
            u = X.solve(X.f)
            dz, dt, _ = X.gradients(u, u, 1.0)
            p = {"u": u, "C": (X.f * u).sum(1), "dz": dz, "dt": dt}
            if kind == "train":  # loss = mean(C + 0.1 V), V = sum of facet area times thickness
                zz, tt = X.z.detach().requires_grad_(True), X.t.detach().requires_grad_(True)
                V = []
                for i in range(len(zz)):
                    XYZ = torch.cat([X.xy, zz[i][:, None]], 1)[X.qc]
                    n = torch.linalg.cross(XYZ[:, 2] - XYZ[:, 0], XYZ[:, 3] - XYZ[:, 1])
                    # the area of a facet projected along its diagonals' normal
                    V.append((0.5 * n.norm(dim=1) * tt[i]).sum())
                V = torch.stack(V)
                V.sum().backward()
                p.update(V=V.detach(), dz=(dz + 0.1 * zz.grad) / len(z),
                         dt=(dt + 0.1 * tt.grad) / len(z))
            parts.append(p)
            del X
        return {k: torch.cat([p[k] for p in parts]) for k in parts[0]}
    if kind == "serve":
        us, Cs, dzs = [], [], []
        for m in _serve_meshes(case, seed):
            X = _Exact(m, _dev(m["xyz"][None, :, 2]), int(round(math.sqrt(len(m["xyz"])))))
            u = X.solve(X.f)
            us.append(u[0]), Cs.append((X.f * u).sum()), dzs.append(X.gradients(u, u, 1.0)[0][0])
        return {"u": torch.cat(us), "C": torch.stack(Cs), "dz": torch.cat(dzs)}
    if kind == "bridge":
        if case["el_per_span"] > 200:  # a sequential factorisation of many blocks
            return None
        m = _bridge(case["el_per_span"], seed)
        X = _Exact(m, _dev(m["xyz"][None, :, 2]), 64)
        u = X.solve(X.f)
        return {"u": u[0], "C": (X.f * u).sum(), "dz": X.gradients(u, u, 1.0)[0][0]}
    if kind == "quads":
        xyz, conn, props = (torch.tensor(a, device=DEV) for a in _loose_quads(case["count"], seed))
        out = [_quad_matrices(xyz[c.long()], p[:, 0], p[:, 1], 0.2)[0]
               for c, p in zip(conn.split(1 << 16), props.split(1 << 16))]
        return torch.cat(out).view(-1, 4, 6, 4, 6).transpose(2, 3).contiguous()
    if kind == "beams":
        xyz, conn, props = (torch.tensor(a, device=DEV) for a in _loose_beams(case["count"], seed))
        return _beam_matrices(xyz[conn.long()], props).view(-1, 2, 6, 2, 6).transpose(2, 3).contiguous()
    row_ptr, col, K, x = _spmv_inputs(case["side"], seed)
    n = len(row_ptr) - 1
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), row_ptr.diff().long())
    y = torch.zeros(n, 6, dtype=torch.float64, device=DEV)
    y.index_add_(0, rows, (K @ x.view(n, 6)[col.long()].unsqueeze(-1)).squeeze(-1))
    return y.view(-1), (x * y.view(-1)).sum().view(1)
