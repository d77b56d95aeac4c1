"""Timed cases of the library's public entry points.

Four kinds of call, each through paper_2604_03411_gb300.binding as a program makes it:

  assemble  one gd_assemble pass: residual, consistent tangent (or the residual alone)
            and updated history of a deformed, partly damaged state;
  solve     one gd_solve of the eliminated Newton system with the tangent of such a state;
  step      one gd_newton_step from a committed state of a load path (gd_set_state,
            gd_newton_step, gd_get_state: the restart loop of a driver program);
  path      one whole load path and the gradient of a loss of its reaction curve
            (gd_set_params, gd_set_state, gd_run_load_path, gd_backward: one iteration
            of a calibration).

Meshes, materials and networks are those of the repository's workloads and tests; sizes
in between and ragged ones come from draw().  Inputs depend on the seed alone.
"""
import numpy as np
import torch

import paper_2604_03411_gb300.binding as B
from paper_2604_03411_gb300 import inputs as I

ENERGY = {"raw": I.ENERGY_ICNN_RAW, "iso": I.ENERGY_ICNN_ISO, "neo": I.ENERGY_NEO_HOOKE}


def listed():
    return [
        # the smallest call: the 8x8 square of the uniaxial study, where launches and
        # host latency count
        dict(name="assemble_square8_fp64", kind="assemble", mesh="square", nx=8, ny=8, nz=0, spec=1, prec="fp64",
             wpsi=16, wyld=8, energy="raw", tangent=True),
        # an ordinary pass: the notched plate of the bench (39,936 Q4) in FP64
        dict(name="assemble_notched_fp64", kind="assemble", mesh="notched", nx=312, ny=128, nz=0, spec=1, prec="fp64",
             wpsi=32, wyld=32, energy="raw", tangent=True),
        # FP64 with the wide networks of the cube study on a ragged 3D block
        dict(name="assemble_block3d_fp64", kind="assemble", mesh="cube", nx=27, ny=26, nz=25, spec=1, prec="fp64",
             wpsi=64, wyld=64, energy="raw", tangent=True),
        # residual-only FP64 pass with the isochoric map and uneven widths (what a user
        # monitors between tangent updates)
        dict(name="residual_block3d_fp64", kind="assemble", mesh="cube", nx=17, ny=16, nz=15, spec=1, prec="fp64",
             wpsi=24, wyld=40, energy="iso", tangent=False),
        # the largest pass: the 64^3 cube of the bench in mixed precision
        dict(name="assemble_cube64_mixed", kind="assemble", mesh="cube", nx=64, ny=64, nz=64, spec=1, prec="mixed",
             wpsi=64, wyld=64, energy="raw", tangent=True),
        # the thin 3D notched plate (2,352 HEX8) in mixed precision: few batches per SM
        dict(name="assemble_plate3d_mixed", kind="assemble", mesh="plate3d", nx=49, ny=48, nz=1, spec=1, prec="mixed",
             wpsi=32, wyld=32, energy="raw", tangent=True),
        # many specimens in one handle (the bench's batch), every one with its own networks
        dict(name="assemble_batch_mixed", kind="assemble", mesh="batch", nx=0, ny=0, nz=0, spec=96, prec="mixed",
             wpsi=0, wyld=0, energy="raw", tangent=True),
        # linear solves: the notched plate's FP64 system, and 3D blocks with FP64 and FP32 values
        dict(name="solve_notched_fp64", kind="solve", mesh="notched", nx=312, ny=128, nz=0, spec=1, prec="fp64",
             wpsi=32, wyld=32, energy="raw"),
        dict(name="solve_block3d_fp64", kind="solve", mesh="cube", nx=33, ny=31, nz=30, spec=1, prec="fp64",
             wpsi=16, wyld=16, energy="raw"),
        dict(name="solve_cube48_mixed", kind="solve", mesh="cube", nx=48, ny=48, nz=48, spec=1, prec="mixed",
             wpsi=16, wyld=16, energy="raw"),
        # forward and backward through a short load path of the square (calibration)
        dict(name="path_square8_fp64", kind="path", mesh="square", nx=8, ny=8, nz=0, spec=1, prec="fp64", wpsi=16,
             wyld=8, energy="raw", steps=12),
        # one FP64 load step of a 3D block whose inner solves run in FP32 and are refined in FP64
        dict(name="step_block3d_refined", kind="step", mesh="cube", nx=32, ny=31, nz=30, spec=1, prec="fp64",
             wpsi=16, wyld=16, energy="raw", steps=2, inner="refined"),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case: the same kinds over the whole range of sizes, widths and options."""
    kind = rng.choice(["assemble", "assemble", "assemble", "assemble", "solve", "solve", "path", "step"])
    w = [8, 16, 24, 32, 40, 48, 64]
    c = dict(kind=kind, spec=1, nz=0, prec=rng.choice(["fp64", "mixed"]), wpsi=rng.choice(w), wyld=rng.choice(w),
             energy=rng.choice(["raw", "raw", "iso", "neo"]))
    if kind == "assemble":
        c["mesh"] = rng.choice(["square", "notched", "cube", "cube", "plate3d", "batch"])
        c["tangent"] = rng.random() < 0.8
        if c["mesh"] in ("square", "notched"):
            e = _log_int(rng, 60, 60000)
            c["nx"] = max(4, int((e * (0.5 + rng.random())) ** 0.5))
            c["ny"] = max(3, e // c["nx"])
        elif c["mesh"] == "cube":
            e = _log_int(rng, 30, 150000 if c["prec"] == "mixed" else 15000)
            n = max(2, round(e ** (1.0 / 3.0)))
            c["nx"], c["ny"] = n + rng.randint(0, 2), n + rng.randint(0, 1)
            c["nz"] = n
        elif c["mesh"] == "plate3d":
            c["nx"], c["ny"], c["nz"] = rng.randint(10, 70), rng.randint(10, 60), 1
        else:
            c["nx"] = c["ny"] = 0
            c["spec"] = rng.randint(2, 96)
            c["energy"] = rng.choice(["raw", "iso"])
            c["wpsi"] = c["wyld"] = 0
    elif kind == "solve":
        c["mesh"] = rng.choice(["square", "notched", "cube"])
        c["wpsi"], c["wyld"], c["energy"] = rng.choice([8, 16]), 8, "raw"
        if c["mesh"] == "cube":
            n = _log_int(rng, 5, 40)
            c["nx"], c["ny"], c["nz"] = n + rng.randint(0, 2), n + rng.randint(0, 1), n
        else:
            e = _log_int(rng, 60, 40000)
            c["nx"] = max(4, int((e * (0.5 + rng.random())) ** 0.5))
            c["ny"] = max(3, e // c["nx"])
    elif kind == "path":
        c.update(prec="fp64", mesh="square", nx=rng.randint(3, 20), ny=rng.randint(3, 16), steps=rng.randint(6, 16),
                 wpsi=rng.choice([8, 16, 32]), wyld=rng.choice([8, 16]), energy=rng.choice(["raw", "iso"]))
    else:
        c.update(prec="fp64", inner=rng.choice(["auto", "refined"]), steps=rng.randint(2, 5), energy="raw",
                 wpsi=rng.choice([16, 32]), wyld=rng.choice([8, 32]))
        mesh = rng.choice(["plate3d", "notched", "cube"])
        if mesh == "plate3d":
            c.update(mesh=mesh, nx=rng.randint(12, 40), ny=rng.randint(10, 36), nz=1)
        elif mesh == "notched":
            c.update(mesh=mesh, nx=rng.randint(30, 150), ny=rng.randint(12, 60))
        else:
            n = rng.randint(5, 20)
            c.update(mesh=mesh, nx=n + rng.randint(0, 2), ny=n + rng.randint(0, 1), nz=n)
    return c


# ---------------------------------------------------------------- problems and states
def _problem(case, seed):
    """The problem (a list of them for a batch): mesh, networks drawn from the seed, material."""
    # a calibration evaluates new networks on every call; elsewhere a program keeps its own
    rng = np.random.default_rng([int(seed) if case["kind"] == "path" else 5, 17])
    if case["mesh"] == "batch":
        out = []
        for i in range(case["spec"]):
            r = np.random.default_rng([17, i])                   # the specimens' sizes are the case's
            nx, ny, w = int(r.integers(16, 97)), int(r.integers(16, 49)), int(r.choice([16, 24, 32]))
            m = I.uniaxial_bc_2d(I.structured_q4(nx, ny, nx / ny, 1.0))
            out.append(I.Problem("s", m, I.icnn_weights(rng, 3, w), I.icnn_weights(rng, 1, w),
                                 I.Material(energy=ENERGY[case["energy"]]), np.array([0.1])))
        return out
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["mesh"] == "square":
        mesh, reach = I.uniaxial_bc_2d(I.structured_q4(nx, ny)), 0.3
    elif case["mesh"] == "notched":
        mesh, reach = I.uniaxial_bc_2d(I.notched_plate_q4(nx, ny)), 0.3
    elif case["mesh"] == "plate3d":
        mesh, reach = I.uniaxial_bc_3d(I.notched_plate_hex8(nx, ny, nz)), 0.25
    else:
        mesh, reach = I.biaxial_bc_3d(I.structured_hex8(nx, ny, nz)), 0.4
    psi, yld = I.icnn_weights(rng, 3, case["wpsi"]), I.icnn_weights(rng, 1, case["wyld"])
    mat = I.Material(energy=ENERGY[case["energy"]])
    if case["energy"] == "neo":
        mat.lambda_e = 5.0
    n = case.get("steps", 1)
    if case["kind"] == "path":                                   # load, unload, reload further
        up = max(2, n // 2)
        down = max(1, n // 4)
        load = I.piecewise_path([0.0, reach, 0.6 * reach, 1.1 * reach], [up, down, max(1, n - up - down)])
    else:
        s = 0.09 + 0.02 * np.random.default_rng([int(seed), 41]).random()
        load = np.linspace(0.0, s * reach * (n + 2), n + 3)[1:]
    return I.Problem("case", mesh, psi, yld, mat, load)


_kept = {}


def _handle(case, prob):
    """The handle of the case's mesh and networks (a program keeps it across states)."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _kept:
        _kept.clear()
        o = B.gd_default_options(precision=B.GD_FP64 if case["prec"] == "fp64" else B.GD_MIXED)
        _kept[key] = B.gd_create_batch(prob, o) if isinstance(prob, list) else B.gd_create(prob, o)
    return _kept[key]


def _edge(mesh):
    """Shortest edge of the elements at every node: the scale of a nodal disturbance."""
    x, c = mesh.coords, mesh.conn
    pairs = [(0, 1), (1, 2), (2, 3), (3, 0)]
    if c.shape[1] == 8:
        pairs += [(a + 4, b + 4) for a, b in pairs] + [(a, a + 4) for a in range(4)]
    le = np.min([np.sqrt(((x[c[:, a]] - x[c[:, b]]) ** 2).sum(1)) for a, b in pairs], axis=0)
    h = np.full(mesh.n_nodes, np.inf)
    for a in range(c.shape[1]):
        np.minimum.at(h, c[:, a], le)
    return h


def _state(prob, seed, converged=False):
    """dofs [n, ndof] and history [n_elems, nq] of a state in the middle of a Newton
    iteration: a stretch of up to 10 % with nodal disturbances of 5 % of the element size;
    damage driven above the history in most elements (loading), a quarter of them
    unloading from a higher one, none within rounding of the switch between the two.
    converged: a smooth state near equilibrium instead, loading everywhere."""
    probs = prob if isinstance(prob, list) else [prob]
    rng = np.random.default_rng([int(seed), 29])
    ds, ks = [], []
    for p in probs:
        m = p.mesh
        d = np.empty((m.n_nodes, m.ndof))
        if converged:
            A = np.diag([rng.uniform(0.04, 0.08)] + [-rng.uniform(0.01, 0.02)] * (m.dim - 1))
            d[:, :m.dim] = m.coords @ A
            d[:, m.dim] = 0.1 + 0.02 * np.sin(3.0 * m.coords[:, 0] + rng.uniform(0.0, 3.0))
            ds.append(d.ravel())
            ks.append(rng.uniform(0.04, 0.06, m.n_elems * m.nq))
            continue
        A = rng.uniform(-0.03, 0.03, (m.dim, m.dim)) + np.diag(rng.uniform(0.03, 0.1, m.dim))
        d[:, :m.dim] = m.coords @ A + 0.05 * _edge(m)[:, None] * rng.uniform(-1.0, 1.0, (m.n_nodes, m.dim))
        d[:, m.dim] = rng.uniform(0.15, 0.3, m.n_nodes)
        unloading = rng.random((m.n_elems, 1)) < 0.25
        ds.append(d.ravel())
        ks.append(np.where(unloading, rng.uniform(0.8, 1.2, (m.n_elems, m.nq)),
                           rng.uniform(0.0, 0.1, (m.n_elems, m.nq))).ravel())
    return np.concatenate(ds), np.concatenate(ks)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _smooth(mesh):
    """A smooth field that vanishes on the boundary box, zero on the prescribed dofs."""
    lo, hi = mesh.coords.min(0), mesh.coords.max(0)
    s = np.ones(mesh.n_nodes)
    for k in range(mesh.dim):
        s = s * np.sin(np.pi * (mesh.coords[:, k] - lo[k]) / (hi[k] - lo[k]))
    x = np.empty((mesh.n_nodes, mesh.ndof))
    for c in range(mesh.ndof):
        x[:, c] = s * (1.0 + 0.3 * c) * np.cos(0.7 * c + mesh.coords[:, 0])
    x[mesh.bc_node, mesh.bc_comp] = 0.0
    return x.ravel()


def _amplitude(seed):
    return 1.0 + 0.5 * np.random.default_rng([int(seed), 31]).random()


def prepare(case, seed):
    prob = _problem(case, seed)
    st = dict(case=case)
    if case["kind"] in ("assemble", "solve"):
        h = _handle(case, prob)
        d, k = _state(prob, seed, case["kind"] == "solve")
        st.update(h=h, d=_dev(d), k=_dev(k))
        vt = torch.float64 if case["prec"] == "fp64" else torch.float32
        nnz = B.gd_csr_pattern(h)[1].size if "nnz" not in h.meta else h.meta["nnz"]
        h.meta["nnz"] = nnz
        if case["kind"] == "assemble":
            st.update(R=torch.empty_like(st["d"]), k1=torch.empty_like(st["k"]),
                      vals=torch.empty(nnz, dtype=vt, device="cuda") if case["tangent"] else None,
                      load=torch.empty(k.size, dtype=torch.int8, device="cuda") if case["prec"] == "fp64" else None)
            return st
        # K x = b for a known x: the tangent at the state, b = K x with prescribed dofs eliminated
        vals = torch.empty(nnz, dtype=vt, device="cuda")
        B.gd_assemble(h, st["d"], st["k"], torch.empty_like(st["d"]), vals, None, None, B.GD_ASM_TANGENT)
        m = prob.mesh
        rowptr, colidx = B.gd_csr_pattern(h)
        n = d.size
        x = _smooth(m) * _amplitude(seed)
        K = torch.sparse_csr_tensor(_dev(rowptr.astype(np.int64)), _dev(colidx.astype(np.int64)), vals.double(),
                                    size=(n, n))
        b = (K @ _dev(x)[:, None])[:, 0]
        b[_dev(m.bc_node.astype(np.int64) * m.ndof + m.bc_comp)] = 0.0
        st.update(vals=vals, b=b, x=torch.empty_like(b))
        return st
    if case["kind"] == "path":
        h = B.gd_create(prob, B.gd_default_options())
        rng = np.random.default_rng([int(seed), 37])
        st.update(h=h, psi=_dev(prob.psi.params), yld=_dev(prob.yld.params), g=rng.uniform(0.5, 1.5, prob.load.size),
                  d0=np.zeros(prob.mesh.n_nodes * prob.mesh.ndof), k0=np.zeros((prob.mesh.n_elems, prob.mesh.nq)))
        return st
    # step: the committed state after `steps` load steps
    inner = B.GD_INNER_REFINED if case["inner"] == "refined" else B.GD_INNER_AUTO
    h = B.gd_create(prob, B.gd_default_options(inner_solve=inner))
    for _ in range(case["steps"]):
        B.gd_newton_step(h)
    d, dp, k, nxt, dpp = B.gd_get_state(h)
    st.update(h=h, d=d, dp=dp, k=k, next=nxt, dpp=dpp if nxt >= 2 else None)
    return st


def run(state):
    case, h = state["case"], state["h"]
    if case["kind"] == "assemble":
        B.gd_assemble(h, state["d"], state["k"], state["R"], state["vals"], state["k1"], state["load"],
                      B.GD_ASM_TANGENT if case["tangent"] else B.GD_ASM_RESIDUAL)
        if case["prec"] == "fp64":
            return state["R"], state["vals"], state["k1"], state["load"]
        # GD_MIXED evaluates every element row and local update in FP32; its FP64 buffers only
        # hold sums of those, so a program takes them on as the FP32 results that they are
        return state["R"].float(), state["vals"], state["k1"].float()
    if case["kind"] == "solve":
        B.gd_solve(h, state["b"], state["x"], state["vals"])
        return state["x"]
    if case["kind"] == "path":
        B.gd_set_params(h, state["psi"], state["yld"])
        B.gd_set_state(h, state["d0"], state["k0"], 0)
        reac, _ = B.gd_run_load_path(h)
        return reac, B.gd_backward(h, state["g"])
    B.gd_set_state(h, state["d"], state["k"], state["next"], dofs_prev=state["dp"], dofs_prev2=state["dpp"])
    rep = B.gd_newton_step(h)
    d, _, k, _, _ = B.gd_get_state(h)
    return rep.reaction, d, k


# ---------------------------------------------------------------- work
def work(case):
    """Inputs read once, outputs written once.  Operations of one assembly pass per
    quadrature point: the energy network with gradient and Hessian (10 w^2 + 40 w), two
    yield-network evaluations (4 w^2 + 20 w each), 8 nd^2 for the tangent; a path or step
    counts two passes and one product with the tangent per load step, a solve one product."""
    probs = _problem(case, 1)
    probs = probs if isinstance(probs, list) else [probs]
    by = fl = nnz_b = sol_f = 0.0
    vb = 8 if case["prec"] == "fp64" else 4
    tangent = case.get("tangent", True)
    for p in probs:
        m, w, y = p.mesh, p.psi.width if case["energy"] != "neo" else 0, p.yld.width
        nd, ndof, qp = m.nen * m.ndof, m.ndof, m.n_elems * m.nq
        if case["mesh"] in ("cube", "plate3d"):
            nx, ny, nz = case["nx"], case["ny"], case["nz"]
            nnz = ndof * ndof * (3 * nx + 1) * (3 * ny + 1) * (3 * nz + 1)
        else:
            nx = int(m.conn[0, 3] - m.conn[0, 0]) - 1
            nnz = ndof * ndof * (3 * nx + 1) * (3 * (m.n_elems // nx) + 1)
        by += m.n_elems * m.nen * 4 + m.n_nodes * (m.dim + 2 * ndof) * 8 + qp * 16 + (nnz * vb if tangent else 0)
        fl += qp * (10 * w * w + 40 * w + 2 * (4 * y * y + 20 * y) + (8 * nd * nd if tangent else 0))
        nnz_b += nnz * vb + nnz / ndof * 4 + 2 * m.n_nodes * ndof * 8
        sol_f += 2 * nnz
    if case["kind"] == "assemble":
        return {"bytes": by, "flops": fl}
    if case["kind"] == "solve":
        return {"bytes": nnz_b, "flops": sol_f}
    n = case["steps"] * 2 if case["kind"] == "path" else 1
    return {"bytes": n * (2 * by + nnz_b), "flops": n * (2 * fl + sol_f)}


# ---------------------------------------------------------------- the same in 64 bits
def _net(p, n_in, w):
    out, at = [], 0
    for shape in ((w, n_in), (w,), (w, w), (w, n_in), (w,), (w,), (n_in,)):
        n = int(np.prod(shape))
        out.append(_dev(np.asarray(p[at:at + n]).reshape(shape)))
        at += n
    return out


def _sp(v):
    return torch.logaddexp(v, torch.zeros((), dtype=v.dtype, device=v.device))


def _net_value(net, x):
    W1, b1, W2, A2, b2, w3, a3 = net
    return _sp(_sp(x @ W1.T + b1) @ W2.T + x @ A2.T + b2) @ w3 + x @ a3


class _Law:
    """The constitutive law of a problem on batches of points, FP64, derivatives by torch's autograd."""

    def __init__(self, p):
        self.m = p.mat
        self.psi = _net(p.psi.params, 3, p.psi.width)
        self.yld = _net(p.yld.params, 1, p.yld.width)
        if self.m.energy != I.ENERGY_NEO_HOOKE:
            z = torch.zeros(1, 3, dtype=torch.float64, device="cuda", requires_grad=True)
            N = _net_value(self.psi, z)
            g = torch.autograd.grad(N.sum(), z)[0][0]
            self.N0 = N.item()
            self.n = (2 * g[0] + 4 * g[1] + g[2]).item() if self.m.energy == I.ENERGY_ICNN_RAW else g[2].item()
        z = torch.zeros(1, 1, dtype=torch.float64, device="cuda", requires_grad=True)
        N = _net_value(self.yld, z)
        self.G0, self.Gs = N.item(), 1.0 / torch.autograd.grad(N.sum(), z)[0].item()

    def G(self, q):
        return self.Gs * (_net_value(self.yld, q[:, None]) - self.G0)

    def psi_e(self, H):
        m = self.m
        Am = H + H.transpose(1, 2) + H.transpose(1, 2) @ H
        tA, AA = Am.diagonal(dim1=1, dim2=2).sum(1), (Am * Am.transpose(1, 2)).sum((1, 2))
        tH, HH = H.diagonal(dim1=1, dim2=2).sum(1), (H * H.transpose(1, 2)).sum((1, 2))
        dH = (H[:, 0] * torch.linalg.cross(H[:, 1], H[:, 2])).sum(1)
        x1, x2, x3 = tA, 2 * tA + 0.5 * (tA * tA - AA), tH + 0.5 * (tH * tH - HH) + dH
        J = 1 + x3
        if m.energy == I.ENERGY_NEO_HOOKE:
            L = torch.log1p(x3)
            return 0.5 * m.mu_e * x1 - m.mu_e * L + 0.5 * m.lambda_e * L * L
        if m.energy == I.ENERGY_ICNN_ISO:
            L = torch.log1p(x3)
            x1, x2 = (3 * torch.expm1(-2 / 3 * L) + x1 * torch.exp(-2 / 3 * L),
                      3 * torch.expm1(3 * torch.log1p(x2 / 3) - 4 * L))
        N = _net_value(self.psi, torch.stack([x1, x2, x3], 1))
        return m.mu_e * (N - self.N0 - self.n * x3) + m.lambda_e * (x3 * x3 / J) ** 2

    def f_d(self, kap):
        return torch.exp(-self.m.eta_d * torch.clamp(kap - self.m.kappa_d, min=0.0))

    def Phi(self, pe, phi, kap):
        m = self.m
        return self.G(pe + m.gamma_d * m.beta_d / m.eta_d * (phi - kap) / self.f_d(kap)) - kap

    def update(self, pe, phi, kn):
        """kappa_{n+1} and the loading flag: the root of Phi above kappa_n where Phi(kappa_n) > 0."""
        load = self.Phi(pe, phi, kn) > 0
        lo, hi = kn.clone(), kn + 1e-2
        for _ in range(12):
            up = self.Phi(pe, phi, hi) > 0
            lo = torch.where(up, hi, lo)
            if not bool((up & load).any()):
                break
            hi = torch.where(up, kn + 2 * (hi - kn), hi)
        k = 0.5 * (lo + hi)
        for it in range(60):
            k = k.detach().requires_grad_(True)
            r = self.Phi(pe, phi, k)
            dr = torch.autograd.grad(r.sum(), k)[0]
            r, k = r.detach(), k.detach()
            lo, hi = torch.where(r > 0, k, lo), torch.where(r > 0, hi, k)
            new = k - r / dr
            ok = (new > lo) & (new < hi) & torch.isfinite(new)
            new = torch.where(ok, new, torch.where((r / dr).abs() < 1e-15, k, 0.5 * (lo + hi)))
            done = (((new - k).abs() <= 1e-15 * torch.clamp(k.abs(), min=1.0)) | ~load).all()
            k = new
            if bool(done):
                break
        return torch.where(load, k, kn), load

    def points(self, H, g, phi, kn, tangent):
        """(P|Y vector|-Y) [n, 13], its total derivative [n, 13, 13] (or None), kappa, loading."""
        with torch.no_grad():
            pe = self.psi_e(H)
        kap, load = self.update(pe, phi, kn)
        v = torch.cat([H.reshape(-1, 9), g, phi[:, None], kap[:, None]], 1).detach().requires_grad_(True)
        m = self.m
        Hv, gv, pv, kv = v[:, :9].reshape(-1, 3, 3), v[:, 9:12], v[:, 12], v[:, 13]
        pe = self.psi_e(Hv)
        F = Hv + torch.eye(3, dtype=torch.float64, device="cuda")
        # adjugate of F^T over J: h = F^-T g without a solver
        cof = torch.stack([torch.linalg.cross(F[:, 1], F[:, 2]), torch.linalg.cross(F[:, 2], F[:, 0]),
                           torch.linalg.cross(F[:, 0], F[:, 1])], 1)
        J = (F[:, 0] * cof[:, 0]).sum(1)
        h = (cof @ gv[:, :, None])[:, :, 0] / J[:, None]
        W = self.f_d(kv) * pe + 0.5 * m.c_d * (h * h).sum(1) + 0.5 * m.beta_d * (pv - kv) ** 2
        s = torch.autograd.grad(W.sum(), v, create_graph=tangent)[0]
        if not tangent:
            return s[:, :13].detach(), None, kap, load
        M = torch.stack([torch.autograd.grad(s[:, i].sum(), v, retain_graph=True)[0] for i in range(13)], 1)
        dPhi = torch.autograd.grad(self.Phi(pe, pv, kv).sum(), v)[0]
        dk = torch.where(load[:, None], -dPhi[:, :13] / dPhi[:, 13:], torch.zeros_like(dPhi[:, :13]))
        return s[:, :13].detach(), M[:, :, :13] + M[:, :, 13:] * dk[:, None, :], kap, load


def _exact_assembly(p, d, kn, tangent, chunk=4096):
    """(R [n_dofs], CSR values or None, kappa [n_elems nq]) of one specimen on the GPU in FP64."""
    m, law = p.mesh, _Law(p)
    dim, ndof, nen = m.dim, m.ndof, m.nen
    nd = nen * ndof
    X, conn = _dev(m.coords), _dev(m.conn.astype(np.int64))
    sg = np.array([[-1, -1, -1], [1, -1, -1], [1, 1, -1], [-1, 1, -1], [-1, -1, 1], [1, -1, 1], [1, 1, 1],
                   [-1, 1, 1]], float)[:nen, :dim]
    xi = np.array([[(q >> k & 1) * 2 - 1 for k in range(dim)] for q in range(nen)], float) / np.sqrt(3.0)
    f = 0.5 * (1 + sg[None] * xi[:, None])                       # [q, a, k]
    N = _dev(f.prod(2))
    dN = _dev(np.stack([0.5 * sg[None, :, k] * np.delete(f, k, 2).prod(2) for k in range(dim)], 2))
    R = torch.zeros(m.n_nodes * ndof, dtype=torch.float64, device="cuda")
    kap = torch.empty(m.n_elems, nen, dtype=torch.float64, device="cuda")
    vals = pos = None
    if tangent:
        key = (conn[:, :, None] * m.n_nodes + conn[:, None, :]).reshape(-1)
        uniq, inv = torch.unique(key, return_inverse=True)
        cnt = torch.bincount(uniq // m.n_nodes, minlength=m.n_nodes)
        first = torch.cumsum(cnt, 0) - cnt                       # blocks before each node's rows
        row = uniq // m.n_nodes
        base = (first * ndof * ndof)[row] + (torch.arange(uniq.numel(), device="cuda") - first[row]) * ndof
        step = (cnt * ndof)[row]                                 # row length
        pos = (base[inv].reshape(-1, nen, nen), step[inv].reshape(-1, nen, nen))
        vals = torch.zeros(int(uniq.numel()) * ndof * ndof, dtype=torch.float64, device="cuda")
    d2 = _dev(d).reshape(-1, ndof)
    kn = _dev(kn).reshape(m.n_elems, nen)
    io = torch.arange(ndof, device="cuda")
    for e0 in range(0, m.n_elems, chunk):
        c = conn[e0:e0 + chunk]
        ne = c.shape[0]
        Jm = torch.einsum("eaj,qak->eqjk", X[c], dN)
        grad = torch.einsum("qak,eqkj->eqaj", dN, torch.linalg.inv(Jm))
        Jw = torch.linalg.det(Jm)
        de = d2[c]
        Bm = torch.zeros(ne, nen, 13, nen, ndof, dtype=torch.float64, device="cuda")
        for i in range(dim):
            for j in range(dim):
                Bm[:, :, 3 * i + j, :, i] = grad[..., j]
        for j in range(dim):
            Bm[:, :, 9 + j, :, dim] = grad[..., j]
        Bm[:, :, 12, :, dim] = N[None]
        Bm = Bm.reshape(ne * nen, 13, nd)
        z = (Bm.reshape(ne, nen * 13, nd) @ de.reshape(ne, nd, 1)).reshape(ne * nen, 13)
        s, M, k1, _ = law.points(z[:, :9].reshape(-1, 3, 3), z[:, 9:12], z[:, 12], kn[e0:e0 + chunk].reshape(-1),
                                 tangent)
        kap[e0:e0 + chunk] = k1.reshape(ne, nen)
        s = s * Jw.reshape(-1, 1)
        Re = (Bm.transpose(1, 2) @ s[:, :, None]).reshape(ne, nen, nd).sum(1)
        R.index_add_(0, (c[:, :, None] * ndof + io).reshape(-1), Re.reshape(-1))
        if tangent:
            Ke = (Bm.transpose(1, 2) @ (M * Jw.reshape(-1, 1, 1)) @ Bm).reshape(ne, nen, nd, nd).sum(1)
            Ke = Ke.reshape(ne, nen, ndof, nen, ndof)
            b, st = pos[0][e0:e0 + chunk], pos[1][e0:e0 + chunk]
            at = b[:, :, None, :, None] + io[None, None, :, None, None] * st[:, :, None, :, None] + io
            vals.index_add_(0, at.reshape(-1), Ke.reshape(-1))
    return R, vals, kap.reshape(-1)


def _exact_path(p):
    """Reactions of every load step by Newton's method with a dense direct solver."""
    m = p.mesh
    n = m.n_nodes * m.ndof
    fixed = np.zeros(n, bool)
    bc = m.bc_node.astype(np.int64) * m.ndof + m.bc_comp
    fixed[bc] = True
    free = _dev(np.nonzero(~fixed)[0])
    conn = m.conn.astype(np.int64)
    pairs = np.unique((conn[:, :, None] * m.n_nodes + conn[:, None, :]).ravel())
    rows, cols = [], []
    for node in range(m.n_nodes):
        nb = pairs[np.searchsorted(pairs, node * m.n_nodes):np.searchsorted(pairs, (node + 1) * m.n_nodes)] % m.n_nodes
        cl = (nb[:, None] * m.ndof + np.arange(m.ndof)).ravel()
        for i in range(m.ndof):
            rows.append(np.full(cl.size, node * m.ndof + i))
            cols.append(cl)
    at = _dev(np.concatenate(rows) * n + np.concatenate(cols))
    rd = _dev(m.react_node.astype(np.int64) * m.ndof + m.react_comp)
    d, kn, out = np.zeros(n), np.zeros(m.n_elems * m.nq), []
    prev, l1, l0 = None, 0.0, 0.0
    for load in p.load:
        if prev is None:
            t = load / (m.coords[:, 0].max() - m.coords[:, 0].min())
            w = d.copy()
            w[0::m.ndof] = m.coords[:, 0] * t
        else:
            w = d + (d - prev) * ((load - l1) / (l1 - l0))
        w[bc] = m.bc_scale * load
        for _ in range(40):
            R, v, k1 = _exact_assembly(p, w, kn, True)
            K = torch.zeros(n * n, dtype=torch.float64, device="cuda")
            K[at] = v
            K = K.reshape(n, n)[free][:, free]
            dx = torch.linalg.solve(K, -R[free])
            w[free.cpu().numpy()] += dx.cpu().numpy()
            if float(dx.abs().max()) < 1e-13:
                break
        R, _, k1 = _exact_assembly(p, w, kn, False)
        out.append(float(R[rd].sum()))
        prev, d, kn, l0, l1 = d, w.copy(), k1.cpu().numpy(), l1, load
    return np.array(out)


def exact(case, seed):
    prob = _problem(case, seed)
    if case["kind"] == "assemble":
        d, k = _state(prob, seed)
        probs = prob if isinstance(prob, list) else [prob]
        parts, dn, kn = [], 0, 0
        for p in probs:
            n, q = p.mesh.n_nodes * p.mesh.ndof, p.mesh.n_elems * p.mesh.nq
            parts.append(_exact_assembly(p, d[dn:dn + n], k[kn:kn + q], case["tangent"]))
            dn, kn = dn + n, kn + q
        R, v, k1 = (torch.cat(x) if x[0] is not None else None for x in zip(*parts))
        return (R, v, k1, None) if case["prec"] == "fp64" else (R, v, k1)
    if case["kind"] == "solve":
        return _dev(_smooth(prob.mesh) * _amplitude(seed))
    if case["kind"] == "path":
        return _exact_path(prob), None
    return None
