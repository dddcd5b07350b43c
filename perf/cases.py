"""What a user of this library has it do, as cases that can be timed and compared.

Each case is one call, or one step of a program, through the public binding
(``paper_2309_05965_gb300.kfbi``): a box solve, one application of the boundary
integral operator, a whole GMRES solve with evaluation, a batch of solves, a
time step of a moving interface, or a training step of the warm-start network.
Data are smooth manufactured fields (sums of seeded plane waves), made on the
GPU.
"""
import math

import numpy as np
import torch

from paper_2309_05965_gb300 import kfbi, learned

F64 = torch.float64
LS_ELLIPSE, LS_STAR, LS_ELLIPSOID, LS_TORUS, LS_MOLECULE, LS_SPHERES, LS_GRID, LS_UNION = 1, 2, 3, 4, 5, 7, 8, 9

# shape -> (dim, half width of the box, level-set kind, problem kind)
SHAPES = {
    "ellipse": (2, 1.0, LS_ELLIPSE, kfbi.DIRICHLET_INTERIOR),
    "ellipse_neumann": (2, 1.0, LS_ELLIPSE, kfbi.NEUMANN_INTERIOR),
    "star": (2, 1.0, LS_STAR, kfbi.INTERFACE_MU),
    "star_general": (2, 1.0, LS_STAR, kfbi.INTERFACE_GENERAL),
    "touching": (2, 1.7, LS_UNION, kfbi.INTERFACE_MU),
    "torus": (3, 1.0, LS_TORUS, kfbi.DIRICHLET_INTERIOR),
    "torus_neumann": (3, 1.5, LS_TORUS, kfbi.NEUMANN_INTERIOR),
    "ellipsoid": (3, 1.0, LS_ELLIPSOID, kfbi.INTERFACE_MU),
    "molecule": (3, 1.0, LS_MOLECULE, kfbi.DIRICHLET_INTERIOR),
    "spheres": (3, 1.5, LS_SPHERES, kfbi.INTERFACE_GENERAL),
}


def listed():
    return [
        # a small Dirichlet problem from start to end, plain FP64: launches and latency decide
        dict(name="solve-ellipse-64-fp64", op="solve", shape="ellipse", n=64, prec="fp64", kappa=0.0, a=0.6, b=0.4),
        # one operator application of the plain FP64 path on an ordinary 2D grid
        dict(name="apply-star-512-fp64", op="apply", shape="star", n=512, prec="fp64", kappa=0.0, a=0.5, b=0.1, k=5,
             contrast=1000.0),
        # the interface problem with a flower at contrast 1000 that the library is quoted on, mixed precision
        dict(name="solve-star-1024-mixed", op="solve", shape="star", n=1024, prec="mixed", kappa=0.0, a=0.5, b=0.1,
             k=5, contrast=1000.0),
        # the largest 2D box solve both precisions take
        dict(name="box2d-2048-mixed", op="box", dim=2, n=2048, prec="mixed", box="dst", order=4, kappa=0.0),
        # the plain FP64 box solve in 3D, modified Helmholtz
        dict(name="box3d-256-fp64", op="box", dim=3, n=256, prec="fp64", box="dst", order=4, kappa=1.0),
        # the same solve by multigrid
        dict(name="box3d-256-mg-mixed", op="box", dim=3, n=256, prec="mixed", box="mg", order=4, kappa=1.0),
        # one application of the 3D operator in mixed precision: what each GMRES iteration runs
        dict(name="apply-torus-256-mixed", op="apply", shape="torus", n=256, prec="mixed", kappa=1.0, a=0.5, b=0.2),
        # the general system of three nearly touching spheres: two box solves and four traces per application
        dict(name="apply-spheres-256-mixed", op="apply", shape="spheres", n=256, prec="mixed", kappa=0.0, a=0.7),
        # a whole 3D Neumann solve in FP64 on a medium grid
        dict(name="solve-neumann-torus-128-fp64", op="solve", shape="torus_neumann", n=128, prec="fp64", kappa=0.0,
             a=1.0, b=0.4),
        # many uneven 2D problems solved together
        dict(name="batch-stars-64", op="batch", count=64, geom=5965, nmax=1024),
        # one time step of a moving interface: new geometry from grid samples, jump data, solve, evaluation
        dict(name="moving-1024-mixed", op="moving", n=1024, t=0.35, contrast=10.0),
        # one minibatch step of the warm-start network
        dict(name="train-8192", op="train", rows=8192, width=256),
    ]


def _shape_case(rng, op, shapes, nmax3):
    """Shape parameters that the drawn grid resolves (the library refuses the others)."""
    s = rng.choice(shapes)
    dim = SHAPES[s][0]
    c = dict(op=op, shape=s, prec=rng.choice(["fp64", "mixed"]), kappa=0.0)
    if s in ("ellipse", "ellipse_neumann"):
        c.update(n=rng.choice([64, 128, 256, 512, 1024]), a=round(rng.uniform(0.5, 0.75), 4),
                 b=round(rng.uniform(0.35, 0.5), 4), kappa=rng.choice([0.0, 1.0]))
    elif s in ("star", "star_general"):
        c.update(n=rng.choice([256, 512, 1024]), a=round(rng.uniform(0.45, 0.6), 4), b=round(rng.uniform(0.02, 0.1), 4),
                 k=rng.randint(3, 5), contrast=round(10 ** rng.uniform(0.3, 3.0), 3))
    elif s == "touching":
        c.update(n=rng.choice([256, 512, 1024]), contrast=round(rng.uniform(0.3, 1.0), 3))
    elif s == "torus":
        c.update(n=rng.choice([64, 128, 256]), a=round(rng.uniform(0.48, 0.55), 4), b=round(rng.uniform(0.2, 0.24), 4),
                 kappa=rng.choice([0.0, 1.0]))
    elif s == "torus_neumann":
        c.update(n=rng.choice([128, 256]), a=round(rng.uniform(0.9, 1.0), 4), b=round(rng.uniform(0.36, 0.4), 4))
    elif s == "ellipsoid":
        c.update(n=rng.choice([64, 128, 256]), a=round(rng.uniform(0.45, 0.7), 4), b=round(rng.uniform(0.4, 0.6), 4),
                 contrast=10.0)
    elif s == "molecule":
        c.update(n=rng.choice([64, 128]), a=round(rng.uniform(0.38, 0.42), 4), kappa=1.0)
    else:
        c.update(n=rng.choice([128, 256]), a=round(rng.uniform(0.55, 0.7), 4))
    if dim == 3:
        c["n"] = min(c["n"], nmax3)
    return c


def draw(rng):
    op = rng.choice(["box", "box", "apply", "apply", "solve", "solve", "batch", "moving", "train"])
    if op == "box":
        dim = rng.choice([2, 3])
        box = "mg" if rng.random() < 0.25 else "dst"
        n = rng.choice([64, 128, 256, 512, 1024, 2048] if dim == 2 else [32, 64, 128, 256])
        return dict(op=op, dim=dim, n=n, prec=rng.choice(["fp64", "mixed"]) if box == "dst" else "mixed", box=box,
                    order=rng.choice([4, 4, 4, 2]), kappa=rng.choice([0.0, round(rng.uniform(0.1, 10.0), 3)]))
    if op == "apply":
        return _shape_case(rng, op, sorted(SHAPES), 256)
    if op == "solve":
        return _shape_case(rng, op, ["ellipse", "ellipse_neumann", "star", "star_general", "touching", "torus",
                                     "ellipsoid", "molecule"], 64)
    if op == "batch":
        return dict(op=op, count=rng.randint(4, 32), geom=rng.randint(0, 10 ** 6), nmax=rng.choice([256, 512, 1024]))
    if op == "moving":
        return dict(op=op, n=rng.choice([256, 512, 1024]), t=round(rng.uniform(0.0, 1.5), 4),
                    contrast=round(10 ** rng.uniform(0.3, 2.0), 3))
    return dict(op=op, rows=int(round(2 ** rng.uniform(8, 14))), width=rng.choice([64, 128, 256]))


# ---- seeded smooth data -------------------------------------------------------

def _rng(seed, salt=0):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, salt])


class Waves:
    """u(x) = sum_m a_m cos(k_m . x + phi_m), with gradient and Laplacians."""

    def __init__(self, seed, salt, dim, terms=5):
        r = _rng(seed, salt)
        self.k = r.uniform(-2.0, 2.0, (terms, dim))
        self.a = r.standard_normal(terms)
        self.p = r.uniform(0.0, 2.0 * math.pi, terms)

    def _sum(self, axes, f):
        out = None
        for k, a, p in zip(self.k, self.a, self.p):
            arg = sum(float(ki) * x for ki, x in zip(k, axes)) + float(p)
            v = float(a) * f(k, arg)
            out = v if out is None else out + v
        return out

    def u(self, axes):
        return self._sum(axes, lambda k, t: torch.cos(t))

    def lap(self, axes, power=1):
        return self._sum(axes, lambda k, t: (-float(k @ k)) ** power * torch.cos(t))

    def dn(self, axes, normals):
        return self._sum(axes, lambda k, t: -sum(float(ki) * n for ki, n in zip(k, normals)) * torch.sin(t))


def _grid_axes(dim, n, lo, hi):
    x = lo + torch.arange(n + 1, dtype=F64, device="cuda") * ((hi - lo) / n)
    return [x.reshape([-1 if k == j else 1 for k in range(dim)]) for j in range(dim)]


def _grid_data(case, cfg, wi, wo):
    """f and Lap f of both sides and the outer boundary values, on the grid."""
    ax = _grid_axes(cfg.dim, cfg.n, cfg.lo, cfg.hi)
    kin = cfg.kappa * (1.0 if cfg.kind == kfbi.INTERFACE_GENERAL else cfg.sigma_in)
    kout = cfg.kappa_out if cfg.kind == kfbi.INTERFACE_GENERAL else cfg.kappa * cfg.sigma_out
    out = {"f_in": cfg.sigma_in * wi.lap(ax) - kin * wi.u(ax),
           "lapf_in": cfg.sigma_in * wi.lap(ax, 2) - kin * wi.lap(ax)}
    if cfg.kind in (kfbi.INTERFACE_MU, kfbi.INTERFACE_GENERAL):
        out.update(f_out=cfg.sigma_out * wo.lap(ax) - kout * wo.u(ax),
                   lapf_out=cfg.sigma_out * wo.lap(ax, 2) - kout * wo.lap(ax), g_b=wo.u(ax))
    return {k: v.contiguous() for k, v in out.items()}


def _boundary_data(P, cfg, wi, wo):
    """Jumps (or boundary values) at the problem's own boundary points."""
    xyz = torch.empty((P.nb, P.dim), dtype=F64, device="cuda")
    nrm = torch.empty_like(xyz)
    kfbi.kfbi_dof_points(P.handle, xyz, nrm)
    x, n = list(xyz.unbind(1)), list(nrm.unbind(1))
    if cfg.kind == kfbi.DIRICHLET_INTERIOR:
        return {"g1": wi.u(x).contiguous()}
    if cfg.kind == kfbi.NEUMANN_INTERIOR:
        return {"g2": (cfg.sigma_in * wi.dn(x, n)).contiguous()}
    return {"g1": (wi.u(x) - wo.u(x)).contiguous(),
            "g2": (cfg.sigma_in * wi.dn(x, n) - cfg.sigma_out * wo.dn(x, n)).contiguous()}


def _problem(case):
    dim, half, ls, kind = SHAPES[case["shape"]]
    s = case["shape"]
    a, b = case.get("a"), case.get("b")
    kw = {}
    if s.startswith("ellipse"):
        p = [0.0, 0.0, a, b, 0.0] if kind == kfbi.DIRICHLET_INTERIOR else [0.0, 0.0, a, b, -math.pi / 6]
    elif s == "ellipsoid":
        p = [0.0, 0.0, 0.0, a, b, 0.5]
        kw.update(sigma_in=case["contrast"])
    elif s.startswith("star"):
        p = [0.0, 0.0, a, b, float(case["k"])]
        kw.update(sigma_in=case["contrast"])
        if s == "star_general":
            kw.update(sigma_in=1.0, sigma_out=4.0, kappa_out=10.0)
    elif s == "touching":
        p = []
        for m in range(1, 9):
            p += [LS_ELLIPSE, math.cos(m * math.pi / 4), math.sin(m * math.pi / 4), 0.383, 0.383, 0.0]
        p = [9.0] + p + [LS_STAR, 0.0, 0.0, 0.514, 0.514 * 0.2, 5.0]
        kw.update(sigma_in=case["contrast"], sigma_out=3.0)
    elif s.startswith("torus"):
        p = [a, b]
        if kind == kfbi.NEUMANN_INTERIOR:
            kw.update(cos_alpha=0.55)
    elif s == "molecule":
        p = [a, 0.5, 3.0, -0.3, 0.0, 0.0, 0.3, 0.0, 0.0, 0.0, 0.3, 0.1]
    else:
        p = [a, 3.0, 0.5, 0.5, 0.5, -0.5, -0.5, 0.5, 0.5, -0.5, -0.5]
        kw.update(sigma_in=1.0, sigma_out=4.0, kappa_out=10.0)
    return kfbi.Problem(dim, case["n"], -half, half, ls, p, kind, kappa=case["kappa"],
                        precision=kfbi.MIXED if case["prec"] == "mixed" else kfbi.FP64, **kw)


# ---- inputs --------------------------------------------------------------------

def _prepare_box(case, seed):
    dim, n = case["dim"], case["n"]
    P = kfbi.Problem(dim, n, -1.0, 1.0, LS_ELLIPSE if dim == 2 else LS_ELLIPSOID,
                     [0.0, 0.0, 0.6, 0.5, 0.0] if dim == 2 else [0.0, 0.0, 0.0, 0.6, 0.6, 0.6], kfbi.DIRICHLET_INTERIOR,
                     kappa=case["kappa"], order=case["order"],
                     box_solver=kfbi.BOX_MG if case["box"] == "mg" else kfbi.BOX_DST,
                     precision=kfbi.MIXED if case["prec"] == "mixed" else kfbi.FP64)
    return {"P": P, "rhs": _box_rhs(case, seed), "u": torch.zeros(P.grid_shape, dtype=F64, device="cuda")}


def _box_rhs(case, seed):
    """A smooth source, and corrections of either sign next to an interface: what a corrected right-hand side holds."""
    dim, n = case["dim"], case["n"]
    ax = _grid_axes(dim, n, -1.0, 1.0)
    r = sum(x * x for x in ax).sqrt()
    f = Waves(seed, 1, dim).u(ax)
    near = (r - 0.55).abs() < 2.0 / n
    return (f + near * (0.1 * n * n) * Waves(seed, 2, dim).u(ax)).contiguous()


def _prepare_batch(case, seed):
    rng = np.random.default_rng(case["geom"])
    sizes = [n for n in (128, 256, 512, 1024) if n <= case["nmax"]]
    problems, datas, keep = [], [], []
    while len(problems) < case["count"]:
        r0, amp = rng.uniform(0.4, 0.6), rng.uniform(0.0, 0.15)
        k, contrast = int(rng.integers(3, 8)), 10.0 ** rng.uniform(0.0, 3.0)
        n = int(rng.choice(sizes))
        if amp * k * k > 0.02 * n:     # the grid has to resolve the star's tips
            continue
        try:
            P = kfbi.Problem(2, n, -1.0, 1.0, LS_STAR, [0.0, 0.0, r0, amp, float(k)], kfbi.INTERFACE_MU,
                             sigma_in=contrast, precision=kfbi.MIXED, box_rtol=1e-11, box_max_iters=3)
        except kfbi.KfbiError as e:
            if e.status != 2:
                raise
            continue
        i = len(problems)
        wi, wo = Waves(seed, 10 + 2 * i, 2), Waves(seed, 11 + 2 * i, 2)
        t = _grid_data(case, P.cfg, wi, wo)
        t.update(_boundary_data(P, P.cfg, wi, wo))
        problems.append(P)
        keep.append(t)
        datas.append(kfbi.make_data(**t))
    B = kfbi.Batch(problems)

    def flat(sizes):
        """One buffer, each instance's part on a 512-byte boundary."""
        off = np.concatenate([[0], np.cumsum([-(-s // 64) * 64 for s in sizes])])
        buf = torch.zeros(int(off[-1]), dtype=F64, device="cuda")
        return buf, [buf[int(o):int(o) + s] for o, s in zip(off, sizes)]

    xbuf, xs = flat([P.nb for P in problems])
    ubuf, us = flat([(P.n + 1) ** 2 for P in problems])
    us = [u.view(P.grid_shape) for u, P in zip(us, problems)]
    opts = kfbi.GmresOpts(rtol=1e-10, restart=100, max_iter=100, x0=None)
    return {"B": B, "datas": datas, "keep": keep, "xbuf": xbuf, "xs": xs, "ubuf": ubuf, "us": us, "opts": opts}


def _moving_samples(n, t):
    """Node values of a wobbly shape that turns and moves with t."""
    x, y = _grid_axes(2, n, -1.0, 1.0)
    cx, cy = 0.08 * math.sin(2 * t), 0.08 * math.cos(3 * t) - 0.08
    c, s = math.cos(0.6 * t), math.sin(0.6 * t)
    xr, yr = c * (x - cx) + s * (y - cy), -s * (x - cx) + c * (y - cy)
    return ((xr / 0.62) ** 2 + (yr / 0.45) ** 2 + 0.25 * torch.sin(3 * xr) * torch.sin(4 * yr) - 1.0).contiguous()


def _prepare_moving(case, seed):
    n = case["n"]
    shift = 0.02 * float(_rng(seed, 3).uniform(-1.0, 1.0))
    P = kfbi.Problem(2, n, -1.0, 1.0, LS_GRID, [], kfbi.INTERFACE_MU, sigma_in=case["contrast"],
                     precision=kfbi.MIXED, ls_samples=_moving_samples(n, case["t"] - 0.05))
    wi, wo = Waves(seed, 1, 2), Waves(seed, 2, 2)
    return {"P": P, "samples": _moving_samples(n, case["t"] + shift), "wi": wi, "wo": wo,
            "grid": _grid_data(case, P.cfg, wi, wo),
            "opts": kfbi.GmresOpts(rtol=1e-10, restart=100, max_iter=200, x0=None),
            "u": torch.zeros(P.grid_shape, dtype=F64, device="cuda"),
            "mask": torch.zeros(P.grid_shape, dtype=torch.uint8, device="cuda")}


def _train_inputs(case, seed):
    r = _rng(seed, 5)
    rows, width, ni = case["rows"], case["width"], kfbi.WS_FEATURES
    total = rows + rows // 2 + 7
    X = r.standard_normal((total, ni)).astype(np.float32)
    t = np.tanh(X[:, 0] + 0.5 * X[:, 1] * X[:, 2]).astype(np.float32) + 0.1 * X[:, 3]
    order = r.permutation(total)[:rows].astype(np.int32)
    lim1, lim2, lim3 = math.sqrt(6.0 / (ni + width)), math.sqrt(3.0 / width), math.sqrt(6.0 / (width + 1))
    params = np.concatenate([r.uniform(-lim1, lim1, width * ni), 0.1 * r.standard_normal(width),
                             r.uniform(-lim2, lim2, width * width), 0.1 * r.standard_normal(width),
                             r.uniform(-lim3, lim3, width), 0.1 * r.standard_normal(1),
                             0.1 * r.standard_normal(ni)]).astype(np.float32)
    return X, t.astype(np.float32), order, params


def _prepare_train(case, seed):
    X, t, order, params = _train_inputs(case, seed)
    net = learned.WarmStart(width=case["width"], seed=1)
    kfbi.kfbi_mlp_set_affine(net.handle, np.zeros(kfbi.WS_FEATURES), np.ones(kfbi.WS_FEATURES), 0.0, 1.0)
    dev = [torch.from_numpy(v).cuda() for v in (X, t, order, params)]
    return {"net": net, "X": dev[0], "t": dev[1], "order": dev[2], "params": dev[3],
            "loss": torch.zeros(1, dtype=torch.float32, device="cuda"), "grads": torch.zeros_like(dev[3]),
            "y": torch.zeros(X.shape[0], dtype=torch.float32, device="cuda")}


def prepare(case, seed):
    op = case["op"]
    if op == "box":
        return dict(case=case, **_prepare_box(case, seed))
    if op == "batch":
        return dict(case=case, **_prepare_batch(case, seed))
    if op == "moving":
        return dict(case=case, **_prepare_moving(case, seed))
    if op == "train":
        return dict(case=case, **_prepare_train(case, seed))
    P = _problem(case)
    dim = P.dim
    size = P.nb * (2 if P.cfg.kind == kfbi.INTERFACE_GENERAL else 1)
    s = {"case": case, "P": P}
    if op == "apply":
        xyz = torch.empty((P.nb, dim), dtype=F64, device="cuda")
        nrm = torch.empty_like(xyz)
        kfbi.kfbi_dof_points(P.handle, xyz, nrm)
        parts = [Waves(seed, 1 + k, dim).u(list(xyz.unbind(1))) for k in range(size // P.nb)]
        s.update(x=torch.cat(parts).contiguous(), y=torch.zeros(size, dtype=F64, device="cuda"))
        return s
    wi, wo = Waves(seed, 1, dim), Waves(seed, 2, dim)
    keep = _grid_data(case, P.cfg, wi, wo)
    keep.update(_boundary_data(P, P.cfg, wi, wo))
    s.update(keep=keep, data=kfbi.make_data(**keep), x=torch.zeros(size, dtype=F64, device="cuda"),
             u=torch.zeros(P.grid_shape, dtype=F64, device="cuda"),
             opts=kfbi.GmresOpts(rtol=1e-10, restart=100, max_iter=200, x0=None))
    return s


def run(s):
    op = s["case"]["op"]
    if op == "box":
        kfbi.kfbi_box_solve(s["P"].handle, s["rhs"], s["u"])
        return s["u"]
    if op == "apply":
        kfbi.kfbi_apply_operator(s["P"].handle, s["x"], s["y"])
        return s["y"]
    if op == "solve":
        kfbi.kfbi_gmres_solve(s["P"].handle, s["data"], s["opts"], s["x"])
        kfbi.kfbi_evaluate(s["P"].handle, s["data"], s["x"], s["u"])
        return {"density": s["x"], "u": s["u"]}
    if op == "batch":
        s["B"].gmres_solve(s["datas"], s["opts"], s["xs"])
        s["B"].evaluate(s["datas"], s["xs"], s["us"])
        return {"density": s["xbuf"], "u": s["ubuf"]}
    if op == "moving":
        P = s["P"]
        P.update_levelset(LS_GRID, [], s["samples"])
        jumps = _boundary_data(P, P.cfg, s["wi"], s["wo"])
        data = kfbi.make_data(**jumps, **s["grid"])
        x = torch.zeros(P.nb, dtype=F64, device="cuda")
        kfbi.kfbi_gmres_solve(P.handle, data, s["opts"], x)
        kfbi.kfbi_evaluate(P.handle, data, x, s["u"])
        kfbi.kfbi_inside_mask(P.handle, s["mask"])
        return {"u": s["u"], "mask": s["mask"]}
    # a step from given parameters: forward over all rows, loss and gradient of the minibatch, one Adam update
    m = s["net"].handle
    kfbi.kfbi_mlp_set_params(m, s["params"])
    kfbi.kfbi_mlp_forward(m, s["X"], s["y"])
    kfbi.kfbi_mlp_loss_grad(m, s["X"], s["t"], rows=s["order"], loss=s["loss"])
    kfbi.kfbi_mlp_adam(m, 1e-3)
    new = torch.empty_like(s["params"])
    kfbi.kfbi_mlp_get_params(m, new, s["grads"])
    return {"loss": s["loss"], "y": s["y"], "grads": s["grads"], "params": new}


# ---- what a pass cannot do without ------------------------------------------------

def _box_work(dim, n, solves=1.0):
    pts = float(n - 1) ** dim
    # every point read and written once; a sine transform of each axis there and back (half a real FFT of length 2N)
    return 16.0 * pts * solves, 2.0 * dim * pts * 2.5 * math.log2(2 * n) * solves


def _iters(case):
    return {2: 10, 3: 14}[SHAPES[case["shape"]][0]]


def work(case):
    op = case["op"]
    if op == "box":
        b, f = _box_work(case["dim"], case["n"])
    elif op == "apply":
        dim, _, _, kind = SHAPES[case["shape"]]
        b, f = _box_work(dim, case["n"], 2 if kind == kfbi.INTERFACE_GENERAL else 1)
    elif op == "solve":
        dim, _, _, kind = SHAPES[case["shape"]]
        b, f = _box_work(dim, case["n"], (_iters(case) + 2) * (2 if kind == kfbi.INTERFACE_GENERAL else 1))
        b += 8.0 * 6 * (case["n"] + 1.0) ** dim
    elif op == "batch":
        b = f = 0.0
        sizes = [n for n in (128, 256, 512, 1024) if n <= case["nmax"]]
        for n in sizes:
            bb, ff = _box_work(2, n, 16.0 * case["count"] / len(sizes))
            b, f = b + bb, f + ff
    elif op == "moving":
        b, f = _box_work(2, case["n"], 11)
        b += 8.0 * 7 * (case["n"] + 1.0) ** 2
    else:
        rows, w, ni = case["rows"], case["width"], kfbi.WS_FEATURES
        total = rows + rows // 2 + 7
        f = 2.0 * w * (w + ni) * (3 * rows + total)
        b = 4.0 * ((ni + 1) * (rows + total) + 5 * w * (w + ni + 3))
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits ------------------------------------------------------------

def _dst_axis(x, axis):
    """DST-I along one axis (interior values), by the odd extension."""
    z = torch.zeros_like(x.narrow(axis, 0, 1))
    ext = torch.cat([z, x, z, -x.flip(axis)], dim=axis)
    return -0.5 * torch.fft.rfft(ext, dim=axis).imag.narrow(axis, 1, x.shape[axis])


def _exact_box(case, seed):
    dim, n, kt = case["dim"], case["n"], case["kappa"]
    h = 2.0 / n
    inner = tuple(slice(1, n) for _ in range(dim))
    rhs = _box_rhs(case, seed)
    x = rhs[inner]
    for ax in range(dim):
        x = _dst_axis(x, ax)
    s = torch.sin(torch.arange(1, n, dtype=F64, device="cuda") * (math.pi / (2 * n))) ** 2
    S = [s.reshape([-1 if k == j else 1 for k in range(dim)]) for j in range(dim)]
    s1 = sum(S)
    if case["order"] == 2:
        lam = -4.0 * s1 / h ** 2 - kt
    elif dim == 2:
        lam = (-4.0 * s1 + 8.0 / 3.0 * S[0] * S[1]) / h ** 2 - kt * (1.0 - s1 / 3.0)
    else:
        s2 = S[0] * S[1] + S[1] * S[2] + S[2] * S[0]
        lam = (-4.0 * s1 + 8.0 / 3.0 * s2 - 4.0 / 3.0 * S[0] * S[1] * S[2]) / h ** 2 - kt * (1.0 - s1 / 3.0)
    x = x / lam
    for ax in range(dim):
        x = _dst_axis(x, ax) * (2.0 / n)
    u = torch.zeros_like(rhs)
    u[inner] = x
    return u


def _exact_train(case, seed):
    X, t, order, params = _train_inputs(case, seed)
    w, ni = case["width"], kfbi.WS_FEATURES
    X, t, order, p32 = (torch.from_numpy(v).cuda() for v in (X, t, order.astype(np.int64), params))
    X, t = X.double(), t.double()
    sizes = [w * ni, w, w * w, w, w, 1, ni]
    parts = [q.double() for q in torch.split(p32, sizes)]
    # the products with W1, W2, W3 use bfloat16 weights; gradients are those at the rounded weights
    for k in (0, 2, 4):
        parts[k] = torch.split(p32, sizes)[k].bfloat16().double()
    v = torch.cat(parts).requires_grad_(True)
    W1, b1, W2, b2, W3, b3, WL = torch.split(v, sizes)

    def net(x):
        a1 = torch.tanh(x @ W1.view(w, ni).T + b1)
        a2 = torch.tanh(a1 @ W2.view(w, w).T + b2)
        return a2 @ W3 + b3 + x @ WL

    loss = 0.5 * ((net(X[order]) - t[order]) ** 2).mean()
    loss.backward()
    g = v.grad
    new = p32.double() - 1e-3 * g / (g.abs() + 1e-8)
    with torch.no_grad():
        y = net(X)
    return {"loss": loss.detach().reshape(1), "y": y, "grads": g, "params": new}


def exact(case, seed):
    if case["op"] == "box":
        return _exact_box(case, seed)
    if case["op"] == "train":
        return _exact_train(case, seed)
    return None    # a solve's 64-bit value is the library's own FP64 path
