"""What a user of this framework has it do, as cases that can be timed and checked.

Every case goes through the package's public entry points: the operator product
(``Kernel.matvec``), the contact solves (``Kernel.solve``, ``bem_solve_batch``), the
adhesive ramp (``ramp.run``) and the warm-start network (``Fno.forward``,
``Fno.gradients``, ``warmstart.predict``).  Inputs are shaped like the workloads of the
repository's tests and benchmark (sphere, flat punch, self-affine rough surfaces,
coating parameters drawn from the same ranges) and are made on the GPU from the seed.

``exact`` evaluates the same mathematics in plain torch, in 64 bits.
"""
import math

import torch

from paper_1807_01885_gb300 import bem, ramp, warmstart

DEV = "cuda"


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # one operator product of the smallest grid in use (the sphere configuration's
        # size): a call's latency and its launches
        dict(name="product_f32_n64", kind="product", precision="fp32", N=64, body="layer", field="direction"),
        # the training resolution of the warm start, on a rigid base
        dict(name="product_f32_n256", kind="product", precision="fp32", N=256, body="rigid", field="pressure"),
        # the headline product
        dict(name="product_f32_n2048", kind="product", precision="fp32", N=2048, body="layer", field="direction"),
        # the double path at the size of the validation runs
        dict(name="product_f64_n512", kind="product", precision="fp64", N=512, body="layer", field="pressure"),
        # sphere on a coating, N = 64, double, to 1e-10: the smallest solve
        dict(name="sphere_f64_n64", kind="solve", precision="fp64", N=64, shape="sphere", body="layer",
             control="depth"),
        # flat punch on a coating, N = 256, double (a cell of the stiffness sweep)
        dict(name="punch_f64_n256", kind="solve", precision="fp64", N=256, shape="punch", body="layer",
             control="depth"),
        # the headline solve: rough surface, N = 2048, float, force control, to 1e-8
        dict(name="rough_f32_n2048", kind="solve", precision="fp32", N=2048, shape="rough", body="layer",
             control="force"),
        # many rough-surface instances of uneven size in one call
        dict(name="batch_f32", kind="batch", precision="fp32", sizes="128,256,512,1024", count=32),
        # loading and the first pull-off steps of an adhesive sphere on a coating, N = 512
        dict(name="adhesive_f32_n512", kind="ramp", precision="fp32", N=512, load=4, unload=8),
        # warm-start inference on one full-size surface
        dict(name="fno_forward_n2048", kind="forward", B=1, N=2048, width=32, modes=16, layers=4, hidden=64),
        # one training pass (loss and every gradient) of the training set's batch size
        dict(name="fno_gradients_n256", kind="gradients", B=16, N=256, width=32, modes=16, layers=4, hidden=64),
        # warm-start pressures of a batch of surfaces at the training resolution
        dict(name="predict_n256", kind="predict", B=32, N=256, width=32, modes=16, layers=4, hidden=64),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["product", "product", "solve", "solve", "batch", "ramp", "forward", "gradients", "predict"])
    if kind == "product":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind=kind, precision=precision, N=2 ** rng.randint(4, 11), tag=rng.randrange(1000),
                    body=rng.choice(["layer", "rigid", "half-space", "open"]),
                    field=rng.choice(["pressure", "direction"]))
    if kind == "solve":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        N = 2 ** (rng.randint(6, 11) if precision == "fp32" else rng.randint(5, 8))
        shape = rng.choice(["rough", "rough", "sphere", "punch"])
        return dict(kind=kind, precision=precision, N=N, shape=shape, body=rng.choice(["layer", "rigid"]),
                    control="depth" if shape == "punch" else rng.choice(["depth", "force"]), tag=rng.randrange(1000))
    if kind == "batch":
        sizes = rng.choice(["128,256,512,1024", "64,128,256", "256", "32,64,128,256,512"])
        return dict(kind=kind, precision="fp32", sizes=sizes, count=log_int(3, 32), tag=rng.randrange(1000))
    if kind == "ramp":
        precision = rng.choice(["fp32", "fp32", "fp64"])
        return dict(kind=kind, precision=precision, N=2 ** rng.randint(6, 8 if precision == "fp32" else 7),
                    load=rng.randint(1, 4), unload=rng.randint(1, 6), tag=rng.randrange(1000))
    cells = log_int(1 << 12, 1 << (20 if kind == "gradients" else 21))
    modes = rng.choice([4, 8, 12, 16])
    N = min(1024, max(2 * modes, 2 * log_int(16, 512)))
    return dict(kind=kind, B=max(1, min(64, cells // (N * N))), N=N, width=rng.choice([8, 16, 32, 32]), modes=modes,
                layers=rng.randint(1, 4), hidden=rng.choice([16, 32, 64]), tag=rng.randrange(1000))


# ---------------------------------------------------------------------------
# inputs

def _gen(case, seed):
    return torch.Generator(device=DEV).manual_seed(1000003 * int(seed) + 17 * int(case.get("tag", 0)) + 5)


def _uniform(g, lo, hi):
    return lo + (hi - lo) * float(torch.rand((), generator=g, device=DEV, dtype=torch.float64))


def _rough(N, delta, g, hurst=0.7, rms_slope=0.1):
    """Self-affine surface by spectral synthesis: flat spectrum below the roll-off L/8,
    q^-2(1+H) above it; the height f = max(z) - z of the indenter, double."""
    q1 = 2.0 * math.pi * torch.fft.fftfreq(N, d=delta, device=DEV, dtype=torch.float64)
    q = torch.sqrt(q1[None, :] ** 2 + q1[:, None] ** 2)
    qr = 2.0 * math.pi / (N * delta / 8.0)
    amp = torch.clamp(q / qr, min=1.0) ** (-(1.0 + hurst))
    amp[q > math.pi / delta] = 0.0
    amp[0, 0] = 0.0
    z = torch.randn((2, N, N), generator=g, device=DEV, dtype=torch.float64)
    z = torch.fft.ifft2(torch.complex(amp * z[0], amp * z[1])).real
    z = z - z.mean()
    gx = (torch.roll(z, -1, 1) - torch.roll(z, 1, 1)) / (2.0 * delta)
    gy = (torch.roll(z, -1, 0) - torch.roll(z, 1, 0)) / (2.0 * delta)
    z = z * (rms_slope / torch.sqrt((gx * gx + gy * gy).mean()))
    return z.max() - z


def _radius2(N, delta):
    x = (torch.arange(N, device=DEV, dtype=torch.float64) + 0.5) * delta - 0.5 * N * delta
    return x[None, :] ** 2 + x[:, None] ** 2


def _rough_instance(N, g):
    """One instance of the rough-surface workload: coating and load as in its recipe."""
    delta = 1.0 / N
    i = dict(N=N, delta=delta, h=delta * math.exp(_uniform(g, math.log(2.0), math.log(200.0))),
             E1=math.exp(_uniform(g, math.log(0.05), math.log(20.0))), nu1=_uniform(g, 0.2, 0.49), E2=1.0,
             nu2=_uniform(g, 0.2, 0.49))
    i["height"] = _rough(N, delta, g)
    i["force"] = 0.0025 * min(i["E1"] / (1 - i["nu1"] ** 2), i["E2"] / (1 - i["nu2"] ** 2))
    return i


def _material(case, g, delta):
    """Coating (h, E1, nu1) and substrate (E2, nu2) of a product case."""
    h = delta * math.exp(_uniform(g, math.log(2.0), math.log(100.0)))
    E1, nu1, nu2 = math.exp(_uniform(g, math.log(0.1), math.log(4.0))), _uniform(g, 0.2, 0.45), _uniform(g, 0.2, 0.45)
    body = case["body"]
    if body == "rigid":
        return dict(h=h, E1=E1, nu1=nu1, E2=math.inf, nu2=nu2)
    if body in ("half-space", "open"):
        return dict(h=math.inf, E1=E1, nu1=nu1, E2=1.0, nu2=nu2)
    return dict(h=h, E1=E1, nu1=nu1, E2=1.0, nu2=nu2)


def _product_setup(case, seed):
    g = _gen(case, seed)
    N = case["N"]
    delta = 1.0 / N
    m = _material(case, g, delta)
    p = torch.randn((N, N), generator=g, device=DEV, dtype=torch.float64)
    if case["field"] == "pressure":
        p = torch.relu(p)           # a contact pressure: zero on half of the cells
    return delta, m, p.to(_dtype(case))


def _solve_setup(case, seed):
    """(delta, material, dc_mode, height, target, tol) of a solve."""
    g = _gen(case, seed)
    N, shape = case["N"], case["shape"]
    if shape == "rough":
        i = _rough_instance(N, g)
        if case["control"] == "depth":
            i["E1"] = min(i["E1"], 1.0)
        delta, f, target = i["delta"], i["height"], i["force"]
        m = dict(h=i["h"], E1=i["E1"], nu1=i["nu1"], E2=math.inf if case["body"] == "rigid" else i["E2"], nu2=i["nu2"])
        if case["control"] == "depth":
            target = float(f.flatten().kthvalue(max(1, N * N // 50)).values)   # the 2 % bearing height
        dc = bem.BEM_DC_FINITE_PART
    elif shape == "sphere":
        a, R, layer = 0.01 * _uniform(g, 0.9, 1.1), 1.0, case["body"] == "layer"
        delta = 4 * 0.01 / N
        m = dict(h=0.01, E1=4.0 if layer else 1.0, nu1=0.3, E2=1.0 if layer else math.inf, nu2=0.3)
        f = _radius2(N, delta) / (2 * R)
        target = a * a / R if case["control"] == "depth" else 1.5e-6 * _uniform(g, 0.8, 1.2) * m["E1"]
        dc = bem.BEM_DC_ZERO if layer else bem.BEM_DC_FINITE_PART   # a stiff coating: see bem.h on k = 0
    else:
        delta = 1.0
        a = N / 4 * _uniform(g, 0.9, 1.1)
        m = dict(h=a * math.exp(_uniform(g, math.log(0.1), math.log(3.0))),
                 E1=math.exp(_uniform(g, math.log(0.1), math.log(10.0))), nu1=0.3,
                 E2=1.0 if case["body"] == "layer" else math.inf, nu2=0.45)
        f = torch.where(_radius2(N, delta) <= a * a, 0.0, 10.0 * N * delta)
        target = 1e-3 * a
        dc = bem.BEM_DC_ZERO if case["body"] == "layer" else bem.BEM_DC_FINITE_PART
    return delta, m, dc, f.to(_dtype(case)), target, 1e-10 if case["precision"] == "fp64" else 1e-8


def _batch_setup(case, seed):
    g = _gen(case, seed)
    sizes = [int(v) for v in case["sizes"].split(",")]
    out = []
    for b in range(case["count"]):
        i = _rough_instance(sizes[b % len(sizes)], g)
        i["height"] = i["height"].float()
        out.append(i)
    return out


def _ramp_setup(case, seed):
    """An adhesive sphere on a soft coating, Tabor parameter 5 with z0 = delta."""
    g = _gen(case, seed)
    N, R, a = case["N"], 1.0, 0.1 * _uniform(g, 0.95, 1.0)
    delta = 4 * 0.1 / N
    m = dict(h=a / 2, E1=0.2, nu1=0.3, E2=1.0, nu2=0.3)
    es = m["E1"] / (1 - m["nu1"] ** 2)
    dgamma = math.sqrt(125.0 * es * es * delta ** 3 / R)
    d = a * a / R
    depths = [d * (k + 1) / case["load"] for k in range(case["load"])]
    depths += [d * (1 - 0.02 * (k + 1)) for k in range(case["unload"])]
    return delta, m, (_radius2(N, delta) / (2 * R)).to(_dtype(case)), depths, dgamma, \
        1e-8 if case["precision"] == "fp32" else 1e-10


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


NET_PARTS = ("Pw", "Pb", "Rre", "Rim", "Ww", "Wb", "Q1w", "Q1b", "Q2w", "Q2b")


def _net_shapes(c):
    W, m, L, H = c["width"], c["modes"], c["layers"], c["hidden"]
    return dict(Pw=(W, 7), Pb=(W,), Rre=(L, W, W, 2 * m, m), Rim=(L, W, W, 2 * m, m), Ww=(L, W, W), Wb=(L, W),
                Q1w=(H, W), Q1b=(H,), Q2w=(H,), Q2b=(1,))


def _net_params(case, g):
    """Float parameters scaled so that activations stay O(1), in the library's order."""
    out = []
    for part, shape in _net_shapes(case).items():
        if part in ("Rre", "Rim"):
            w = torch.rand(shape, generator=g, device=DEV) / case["width"] ** 2
        else:
            w = torch.randn(shape, generator=g, device=DEV) * (0.05 if part.endswith("b") else shape[-1] ** -0.5)
        out.append(w.reshape(-1))
    return torch.cat(out)


def _net_inputs(case, seed):
    """Surfaces of B samples, their parameters, mean pressures, features and targets."""
    g = _gen(case, seed)
    B, N = case["B"], case["N"]
    w = _net_params(case, g)
    heights = torch.stack([_rough(N, 1.0 / N, g) for _ in range(B)]).float()
    u = torch.rand((B, 4), generator=g, device=DEV, dtype=torch.float64)
    params = torch.stack([torch.exp(math.log(2.0) + math.log(100.0) * u[:, 0]),
                          torch.exp(math.log(0.05) + math.log(400.0) * u[:, 1]), 0.2 + 0.29 * u[:, 2],
                          0.2 + 0.29 * u[:, 3]], 1).contiguous()
    pbar = 1e-3 * (1.0 + torch.rand((B,), generator=g, device=DEV, dtype=torch.float64))
    return w, heights, params, pbar, g


def _features(heights, params):
    """The network's 7 input features, in double (see bem_fno_features)."""
    B, N = heights.shape[0], heights.shape[-1]
    f = heights.double()
    mean = f.mean(dim=(1, 2), keepdim=True)
    x = torch.empty((B, 7, N, N), dtype=torch.float64, device=DEV)
    x[:, 0] = (f - mean) / torch.sqrt(((f - mean) ** 2).mean(dim=(1, 2), keepdim=True))
    x[:, 1] = (torch.log(params[:, 0]) / math.log(200.0))[:, None, None]
    x[:, 2] = (torch.log(params[:, 1]) / math.log(20.0))[:, None, None]
    x[:, 3] = params[:, 2][:, None, None]
    x[:, 4] = params[:, 3][:, None, None]
    at = (torch.arange(N, device=DEV, dtype=torch.float64) + 0.5) / N
    x[:, 5] = at[None, None, :]
    x[:, 6] = at[None, :, None]
    return x


def _targets(case, g):
    """A sparse pressure field of mean 1, as the solver's solutions are."""
    B, N = case["B"], case["N"]
    q = torch.relu(torch.randn((B, N, N), generator=g, device=DEV) - 1.0)
    return (q / q.mean(dim=(1, 2), keepdim=True)).contiguous()


# ---------------------------------------------------------------------------
# the calls

def _net(case, w):
    net = bem.Fno(width=case["width"], modes=case["modes"], layers=case["layers"], hidden=case["hidden"])
    net.set_params(w)
    return net


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "product":
        delta, m, p = _product_setup(case, seed)
        op = bem.BEM_OP_OPEN if case["body"] == "open" else bem.BEM_OP_PERIODIC
        s.update(k=bem.Kernel(case["N"], delta, precision=case["precision"], op_kind=op, **m), p=p,
                 u=torch.empty_like(p))
    elif kind == "solve":
        delta, m, dc, f, target, tol = _solve_setup(case, seed)
        s.update(k=bem.Kernel(case["N"], delta, precision=case["precision"], dc_mode=dc, **m), f=f, target=target,
                 tol=tol, p=torch.empty_like(f))
    elif kind == "batch":
        insts = _batch_setup(case, seed)
        ks = [bem.Kernel(i["N"], i["delta"], i["h"], i["E1"], i["nu1"], i["E2"], i["nu2"],
                         precision=case["precision"]) for i in insts]
        probs = [bem.make_problem(i["height"], bem.BEM_CTRL_FORCE, i["force"], tol=1e-8, max_iter=5000) for i in insts]
        s.update(insts=insts, ks=ks, probs=probs, outs=[torch.empty_like(i["height"]) for i in insts])
    elif kind == "ramp":
        delta, m, f, depths, dgamma, tol = _ramp_setup(case, seed)
        s.update(k=bem.Kernel(case["N"], delta, precision=case["precision"], **m), f=f, depths=depths, dgamma=dgamma,
                 tol=tol)
    else:
        w, heights, params, pbar, g = _net_inputs(case, seed)
        s["net"] = _net(case, w)
        if kind == "predict":
            s.update(heights=heights, params=params, pbar=pbar)
        else:
            s["x"] = _features(heights, params).float()
            if kind == "forward":
                s["out"] = torch.empty_like(heights)
            else:
                s.update(q=_targets(case, g), grad=torch.empty_like(w))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "product":
        return s["k"].matvec(s["p"], s["u"])
    if kind == "solve":
        p, res = s["k"].solve(s["f"], case["control"], s["target"], tol=s["tol"], p_out=s["p"])
        return dict(p=p, force=res["force"], depth=res["depth"])
    if kind == "batch":
        _, res = bem.bem_solve_batch([k.handle for k in s["ks"]], s["probs"], s["outs"])
        return dict(p=s["outs"], depth=[r["depth"] for r in res])
    if kind == "ramp":
        rec, (p, _) = ramp.run(s["k"], s["f"], s["depths"], s["dgamma"], tol=s["tol"], with_state=True)
        return dict(p=p, force=[r["force"] for r in rec])
    if kind == "forward":
        return s["net"].forward(case["B"], case["N"], s["x"], s["out"])
    if kind == "gradients":
        loss = s["net"].gradients(case["B"], case["N"], s["x"], s["q"], s["grad"])
        return dict(loss=loss, grad=s["grad"])
    return warmstart.predict(s["net"], s["heights"], s["params"], s["pbar"], q_min=0.0)


# ---------------------------------------------------------------------------
# work

def _product_flops(N):
    """Two real transforms of N zero-padded rows and two complex ones of N + 1 columns
    (5 L log2 L operations for a complex length L, half of it for a real one)."""
    M = 2 * N
    return 2 * N * 2.5 * M * math.log2(M) + 2 * (N + 1) * 5 * M * math.log2(M)


def _solve_steps(N):
    """Operator products that a solve of this grid takes, roughly."""
    return 42 * (N / 128) ** 0.45


def work(case):
    kind = case["kind"]
    if kind in ("product", "solve", "ramp"):
        N, e = case["N"], 8 if case["precision"] == "fp64" else 4
        once = 2 * e * N * N + e * (N + 1) ** 2          # p or f, u or p, the compliance
        if kind == "product":
            return dict(bytes=once, flops=_product_flops(N))
        n = _solve_steps(N) * (case["load"] + case["unload"] if kind == "ramp" else 1)
        return dict(bytes=once, flops=n * _product_flops(N))
    if kind == "batch":
        sizes = [int(v) for v in case["sizes"].split(",")]
        ns = [sizes[b % len(sizes)] for b in range(case["count"])]
        return dict(bytes=sum(8 * N * N + 4 * (N + 1) ** 2 for N in ns),
                    flops=sum(_solve_steps(N) * _product_flops(N) for N in ns))
    B, N, W, m, L, H = (case[k] for k in ("B", "N", "width", "modes", "layers", "hidden"))
    cells = B * N * N
    pointwise = 2 * (7 * W + L * W * W + H * W + H)
    spectral = 2 * L * W * 2 * 2 * m                     # along y, forward and inverse
    flops = cells * (pointwise + spectral) + L * B * W * (8 * 2 * m * m * W + 16 * N * 2 * m * m)
    weights = 4 * sum(math.prod(v) for v in _net_shapes(case).values())
    if kind == "gradients":
        return dict(bytes=4 * cells * 8 + 2 * weights, flops=3 * flops)
    return dict(bytes=4 * cells * (8 if kind == "forward" else 2) + weights, flops=flops)


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch

def _khat(N, delta, m, dc_mode, body="layer"):
    """Compliance on the rows [0, 2N) x [0, N] of the 2N period's wave numbers."""
    M = 2 * N
    if body == "open":
        off = torch.arange(-(N - 1), N, device=DEV, dtype=torch.float64) * delta
        h, X, Y = 0.5 * delta, off[None, :], off[:, None]

        def F(s, t):
            return s * torch.asinh(t / s.abs()) + t * torch.asinh(s / t.abs())

        G = (F(X + h, Y + h) - F(X + h, Y - h) - F(X - h, Y + h) + F(X - h, Y - h)) \
            * ((1 - m["nu1"] ** 2) / (math.pi * m["E1"]))
        wrap = torch.zeros((M, M), device=DEV, dtype=torch.float64)
        at = torch.arange(-(N - 1), N, device=DEV) % M
        wrap[at[:, None], at[None, :]] = G
        return torch.fft.rfft2(wrap).real
    i = torch.arange(M, device=DEV, dtype=torch.float64)
    i = torch.minimum(i, M - i)
    j = torch.arange(N + 1, device=DEV, dtype=torch.float64)
    k = torch.sqrt(i[:, None] ** 2 + j[None, :] ** 2) * (2 * math.pi / (M * delta))
    k[0, 0] = 1.0
    c = 2 * (1 - m["nu1"] ** 2) / m["E1"]
    if math.isinf(m["h"]):
        K, dc = c / k, 0.0
    else:
        n1, n2 = m["nu1"], m["nu2"]
        if math.isinf(m["E2"]):
            al, be = 1.0, 0.0
        else:
            a, b = m["E2"] * (1 + n1), m["E1"] * (1 + n2)
            al, be = a / (a + b), b / (a + b)
        A = ((3 - 4 * n1) * al - (3 - 4 * n2) * be) * (be - al)
        B = 4 * (al + (3 - 4 * n2) * be) * (be - al)
        C = (4 * n2 - 3) * be ** 2 - 2 * (2 * n1 - 1) * (2 * n2 - 1) * al * be + (8 * n1 ** 2 - 12 * n1 + 5) * al ** 2
        D = (al + (3 - 4 * n2) * be) * ((3 - 4 * n1) * al + be)
        x = k * m["h"]
        e2 = torch.exp(-2 * x)
        K = c / k * (A * e2 * e2 + B * x * e2 + D) / (-A * e2 * e2 - B * x * x * e2 + 2 * C * e2 + D)
        n0, d0 = A + D, -A + 2 * C + D
        dc = c * m["h"] * ((B - 4 * A) * d0 - n0 * (4 * A - 4 * C)) / (d0 * d0)
    K[0, 0] = 0.0 if dc_mode == bem.BEM_DC_ZERO else dc
    return K


def _matvec(K, p):
    N = p.shape[0]
    return torch.fft.irfft2(torch.fft.rfft2(p, s=(2 * N, 2 * N)) * K, s=(2 * N, 2 * N))[:N, :N]


def _contact(K, f, delta, control, target, tol=1e-11, max_iter=3000):
    """Constrained conjugate gradients (p >= 0, gap >= 0, p gap = 0); (p, depth)."""
    force = control == "force"
    f = f.double()
    if force:
        d, p = 0.0, torch.full_like(f, target / (delta * delta * f.numel()))
    else:
        d, q = target, torch.relu(target - f)
        p = q * ((q * (d - f)).sum() / (q * _matvec(K, q)).sum())
    t, G_old, keep, changed = torch.zeros_like(f), 1.0, 0.0, True
    for _ in range(max_iter):
        on = p > 0
        n = on.sum()
        u = _matvec(K, p)
        g = u + f - d
        if force:
            shift = float((g * on).sum() / n)
            g, d = g - shift, d + shift
        G = ((g * on) ** 2).sum()
        if float(torch.sqrt(G / ((u * on) ** 2).sum())) <= tol and not changed:
            return p, d
        t = torch.where(on, g + keep * (G / G_old) * t, 0.0)
        G_old = G
        r = _matvec(K, t)
        if force:
            r = r - (r * on).sum() / n
        tau = (g * t).sum() / (r * t).sum()
        if not bool(tau > 0):
            if keep == 0.0:
                return p, d
            keep = 0.0
            continue
        p = torch.where(on, p - tau * t, p)
        gone = p < 0
        p = torch.relu(p)
        back = (p == 0) & (g < 0) & ~on
        p = torch.where(back, -tau * g, p)
        keep = 0.0 if int(back.sum()) > 0.1 * int(n) else 1.0
        changed = bool(gone.any() | back.any())
        if force:
            p = p * (target / (delta * delta * p.sum()))
    return None


def _adhesive(K, f, delta, depths, sig, tol=1e-12):
    """The displacement-controlled adhesive procedure; (p, forces), None if it cycles."""
    f = f.double()
    C, x, forces = torch.zeros_like(f, dtype=torch.bool), torch.zeros_like(f), []
    for d in depths:
        x = x * C
        for outer in range(1000):
            b = torch.where(C, d - f, 0.0)
            r = b - torch.where(C, _matvec(K, x), 0.0)
            s, rr, bb = r.clone(), (r * r).sum(), float((b * b).sum())
            for _ in range(5000):
                if bb == 0.0 or float(rr) <= tol * tol * bb:
                    break
                q = torch.where(C, _matvec(K, s), 0.0)
                a = rr / (s * q).sum()
                x = x + a * s
                r = r - a * q
                new = (r * r).sum()
                s = r + (new / rr) * s
                rr = new
            pad = torch.zeros((f.shape[0] + 2, f.shape[1] + 2), dtype=torch.bool, device=DEV)
            pad[1:-1, 1:-1] = C
            inner = pad[:-2, 1:-1] & pad[2:, 1:-1] & pad[1:-1, :-2] & pad[1:-1, 2:]
            add = ~C & (_matvec(K, x) + f - d < 0)
            off = C & ~inner & (-x > sig)
            if not bool(add.any() | off.any()):
                break
            C = (C | add) & ~off
            x = x * C
        else:
            return None
        forces.append(float(delta * delta * x.sum()))
    return x, forces


def _net_exact(case, w, x):
    """The network in double with the bfloat16 values of its weights; (out, weights)."""
    P, at = {}, 0
    for part, shape in _net_shapes(case).items():
        n = math.prod(shape)
        P[part] = w[at:at + n].bfloat16().double().reshape(shape).requires_grad_(case["kind"] == "gradients")
        at += n
    N, m = case["N"], case["modes"]
    n = torch.arange(N, device=DEV, dtype=torch.float64)

    def wave(k, sign):
        a = (k[:, None] * n[None, :]) % N * (2 * math.pi / N)
        return torch.complex(torch.cos(a), sign * torch.sin(a))

    ky = torch.arange(m, device=DEV, dtype=torch.float64)
    kx = torch.cat([ky, ky + (N - m)])
    Ey, Ex = wave(ky, -1.0), wave(kx, -1.0)                 # [m, N], [2m, N]
    c = torch.full((m,), 2.0, device=DEV, dtype=torch.float64)
    c[0] = 1.0

    def pw(W, b, v):
        return torch.einsum("oc,bcxy->boxy", W, v) + b[None, :, None, None]

    v = pw(P["Pw"], P["Pb"], x)
    for l in range(case["layers"]):
        A = torch.complex(v @ Ey.real.T, v @ Ey.imag.T)     # [B, W, N, m]
        X = torch.einsum("ax,bcxk->bcak", Ex, A)
        Y = torch.einsum("biak,ioak->boak", X, torch.complex(P["Rre"][l], P["Rim"][l]))
        A = torch.einsum("ax,boak->boxk", Ex.conj(), Y) * (c / (N * N))
        z = A.real @ Ey.real + A.imag @ Ey.imag + pw(P["Ww"][l], P["Wb"][l], v)
        v = torch.nn.functional.gelu(z) if l < case["layers"] - 1 else z
    h = torch.nn.functional.gelu(pw(P["Q1w"], P["Q1b"], v))
    return torch.einsum("c,bcxy->bxy", P["Q2w"], h) + P["Q2b"], P


def exact(case, seed):
    kind = case["kind"]
    if kind == "product":
        delta, m, p = _product_setup(case, seed)
        return _matvec(_khat(case["N"], delta, m, 0, case["body"]), p.double())
    if kind == "solve":
        delta, m, dc, f, target, _ = _solve_setup(case, seed)
        got = _contact(_khat(case["N"], delta, m, dc), f, delta, case["control"], target)
        if got is None:
            return None
        return dict(p=got[0], force=delta * delta * float(got[0].sum()), depth=got[1])
    if kind == "batch":
        ps, ds = [], []
        for i in _batch_setup(case, seed):
            got = _contact(_khat(i["N"], i["delta"], i, 0), i["height"], i["delta"], "force", i["force"], tol=1e-10)
            ps.append(None if got is None else got[0])
            ds.append(None if got is None else got[1])
        return dict(p=ps, depth=ds)
    if kind == "ramp":
        delta, m, f, depths, dgamma, _ = _ramp_setup(case, seed)
        sig = math.sqrt(m["E1"] / (1 - m["nu1"] ** 2) * dgamma / (0.473201 * delta))
        got = _adhesive(_khat(case["N"], delta, m, 0), f, delta, depths, sig)
        return None if got is None else dict(p=got[0], force=got[1])
    w, heights, params, pbar, g = _net_inputs(case, seed)
    if kind == "predict":
        with torch.no_grad():
            parts = [_net_exact(case, w, _features(heights[b:b + 1], params[b:b + 1]))[0] for b in range(case["B"])]
        return torch.relu(torch.cat(parts)) * pbar[:, None, None]
    x = _features(heights, params).float()
    if kind == "forward":
        with torch.no_grad():
            return torch.cat([_net_exact(case, w, x[b:b + 1].double())[0] for b in range(case["B"])])
    q = _targets(case, g)
    loss, grad = 0.0, None
    for b in range(case["B"]):
        out, P = _net_exact(case, w, x[b:b + 1].double())
        part = ((out - q[b:b + 1].double()) ** 2).sum() / q.numel()
        part.backward()
        loss += float(part)
        one = torch.cat([P[k].grad.reshape(-1) for k in NET_PARTS])
        grad = one if grad is None else grad + one
    return dict(loss=loss, grad=grad)
