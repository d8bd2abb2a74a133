"""Performance cases: what users of this framework run, through its public entry points.

Three families:

- "flow": a solver's run. The solver (mesh, operators, workspace, launch
  shapes, gate network) is the plan a program makes once and keeps; a pass
  hands it a new initial state in device memory, advances a number of stages
  and takes the state out. The double-precision form hands on doubles, the
  single-precision form's state is handed on in single precision.
- "items": a queue of states in host memory through the pipelined call.
- "train" and "infer": the troubled-cell gate's network, one optimiser step
  (gradient, then Adam) and the logits of a set of samples.

`exact` is the same method in double precision, in plain torch.
"""
import math

import numpy as np
import torch

from paper_2306_04467_gb300 import gate, gks2l, inputs

_PLAN = {}          # the plan of the last flow or items case, as a program keeps its solver


def listed():
    return [
        # the smallest configuration (unit square, 16 x 16 squares) over a
        # whole run's worth of stages: launches and latency count
        dict(name="smooth_fp64_512", kind="flow", problem="smooth", nx=16, ny=16, precision="fp64", stages=100),
        # validation-sized run of the plain double form: walls, bathymetry
        dict(name="lake_fp64_66k", kind="flow", problem="lake", nx=181, ny=181, precision="fp64", stages=6),
        # an exchange with another program every step, the smallest call
        dict(name="coupled_fp32_4k6", kind="flow", problem="smooth", nx=48, ny=48, precision="fp32", stages=2),
        # ordinary single-precision run, odd size, fits the L2, on a stream of its own
        dict(name="smooth_fp32_32k", kind="flow", problem="smooth", nx=127, ny=127, precision="fp32", stages=40, stream=True),
        # the internal wave over a ridge, plain single precision, beyond the L2
        dict(name="ridge_fp32_1m", kind="flow", problem="ridge", nx=2043, ny=255, precision="fp32", stages=20, stream=True),
        # the same with the troubled-cell gate and tuned launch shapes, as production runs take it
        dict(name="ridge_gated_1m", kind="flow", problem="ridge", nx=2043, ny=255, precision="fp32", stages=20,
             gate=True, tune=True, stream=True),
        # interface dam break with the gate, launch shapes as they come
        dict(name="dambreak_gated_181k", kind="flow", problem="dambreak", nx=301, ny=301, precision="fp32",
             stages=20, gate=True),
        # a batch of independent instances on meshes of uneven size
        dict(name="ensemble_fp32_24", kind="flow", problem="ensemble", instances=24, lo=5000, hi=40000,
             precision="fp32", stages=10),
        # large interface jumps, which run with the positivity option only
        dict(name="circle_positive_12k8", kind="flow", problem="circle", nx=80, ny=80, precision="fp32", stages=40,
             positivity=0.01),
        # a queue of states in host memory, served through the pipelined call
        dict(name="items_fp64_5k", kind="items", problem="channel", nx=100, ny=25, precision="fp64", items=8,
             stages=10),
        # one optimiser step of the gate's training, at its default batch
        dict(name="train_8192", kind="train", n=8192),
        # the gate's logits over a harvested set of samples
        dict(name="infer_1m", kind="infer", n=1000003),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(("fp64", "fp32", "fp32", "gated", "gated", "ensemble", "positive", "items", "train", "infer"))
    if what == "train":
        return dict(kind="train", n=_log(rng, 500, 40000))
    if what == "infer":
        return dict(kind="infer", n=_log(rng, 2000, 1000000))
    if what == "ensemble":
        lo = _log(rng, 2000, 8000)
        return dict(kind="flow", problem="ensemble", instances=rng.randint(3, 24), lo=lo, hi=lo * rng.randint(2, 5),
                    precision="fp32", stages=2 * rng.randint(1, 5))
    if what == "items":
        ny = _log(rng, 12, 40)
        return dict(kind="items", problem="channel", nx=4 * ny + rng.randint(0, 3), ny=ny,
                    precision="fp64", items=rng.randint(2, 8), stages=rng.randint(1, 10))
    if what == "positive":
        n = _log(rng, 24, 160)
        return dict(kind="flow", problem="circle", nx=n, ny=n, precision=rng.choice(("fp32", "fp64")),
                    stages=2 * rng.randint(1, 8), positivity=0.01)
    if what == "fp64":
        ny = _log(rng, 9, 140)
        return dict(kind="flow", problem=rng.choice(("smooth", "lake", "dambreak")), nx=_log(rng, ny, 1.5 * ny),
                    ny=ny, precision="fp64", stages=rng.randint(1, 6))
    ny = _log(rng, 12, 250)
    problem = rng.choice(("smooth", "ridge", "dambreak") + (("lake",) if what == "fp32" else ()))
    nx = _log(rng, 4 * ny, 8 * ny) if problem == "ridge" else _log(rng, ny, 1.5 * ny)
    case = dict(kind="flow", problem=problem, nx=nx, ny=ny, precision="fp32", stages=rng.randint(1, 20))
    if what == "gated":
        case["gate"] = True
    if rng.random() < 0.5:
        case["stream"] = True
    return case


# ------------------------------------------------------------------ problems

_DOMAIN = {"smooth": (0.0, 1.0, 0.0, 1.0), "lake": (0.0, 1.0, 0.0, 1.0), "ridge": (0.0, 8.0, 0.0, 1.0),
           "dambreak": (-1.0, 1.0, -1.0, 1.0), "ensemble": (0.0, 1.0, 0.0, 1.0), "circle": (0.0, 10.0, 0.0, 10.0),
           "channel": (0.0, 1.0, 0.0, 0.25)}
_PERIODIC = ("smooth", "ensemble", "channel")
_CHI = {"ridge": 0.97}


def _bottom(problem, k, x, y):
    if problem == "smooth":
        return 0.1 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y)
    if problem == "lake":
        return 0.5 * np.exp(-50 * ((x - 0.5) ** 2 + (y - 0.5) ** 2))
    if problem == "ridge":
        return 0.3 * np.exp(-20 * (x - 4) ** 2)
    if problem == "channel":
        return 0.5 * np.exp(-100 * (x - 0.5) ** 2)
    if problem == "ensemble":
        return inputs.fourier_bathymetry(2310 + k)(x, y)
    return np.zeros_like(x)


class _Plan:
    """What a program makes once: meshes, bathymetry, the solver."""

    def __init__(self, case):
        self.problem = case["problem"]
        if self.problem == "ensemble":
            sizes = [(int(n), int(n)) for n in inputs.ensemble_sizes(case["instances"], case["lo"], case["hi"])]
        else:
            sizes = [(case["nx"], case["ny"])]
        bc = "periodic" if self.problem in _PERIODIC else "wall"
        self.meshes = [inputs.jittered_mesh(nx, ny, _DOMAIN[self.problem], seed=2306 + k, bc=bc)
                       for k, (nx, ny) in enumerate(sizes)]
        self.b = [inputs.vertex_samples(lambda x, y, k=k: _bottom(self.problem, k, x, y), m)
                  for k, m in enumerate(self.meshes)]
        self.fp32 = case["precision"] == "fp32"
        par = dict(chi=_CHI.get(self.problem, 0.98), cfl=0.5,
                   precision=gks2l.GKS2L_FP32 if self.fp32 else gks2l.GKS2L_FP64)
        if case.get("positivity"):
            par["positivity_floor"] = case["positivity"]
        if case.get("gate"):
            par["indicator"] = gks2l.GKS2L_INDICATOR_MLP
            par["indicator_threshold"] = gate.THRESHOLD
        self.solver = gks2l.Solver(self.meshes, gks2l.default_params(**par), np.concatenate(self.b),
                                   stream=torch.cuda.Stream() if case.get("stream") else None)
        if case.get("gate"):
            self.solver.set_mlp(_network())
        if case.get("tune"):
            first = _state(self, 0)
            self.solver.stream.wait_stream(torch.cuda.current_stream())
            self.solver.set_state_device(*first)
            self.solver.autotune(2)
            self.solver.stream.synchronize()


def _plan(case):
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _PLAN:
        _PLAN.clear()
        _PLAN[key] = _Plan(case)
    return _PLAN[key]


def _network():
    """A troubled-cell network with fixed weights: it adds up, over both
    layers, how far the neighbours' gradients are from the cell's own, and how
    far the interface's averages are apart beyond a quarter of the features'
    norm; a cell is smooth while that is small."""
    P = np.zeros(gks2l.GKS2L_MLP_NPARAM, np.float32)
    W1, b1 = P[:768].reshape(32, 24), P[768:800]
    W2, w3 = P[800:1824].reshape(32, 32), P[1856:1888]
    u = 0
    for layer in range(2):
        for m in (1, 2, 3):
            for d in (1, 2):
                for sign in (1.0, -1.0):
                    W1[u, 12 * layer + 3 * m + d] = sign
                    W1[u, 12 * layer + d] = -sign
                    u += 1
    for m in (1, 2, 3):
        for sign in (1.0, -1.0):
            W1[u, 3 * m] = 4.0 * sign
            b1[u] = -1.0
            u += 1
    W2[np.arange(u), np.arange(u)] = 1.0
    w3[:u] = 20.0
    P[1888] = -6.0
    P[1889 + 24:] = 1.0
    return P


def _modes(mesh, periodic, seed):
    """Four smooth modes of the domain with random phases: averages over the
    cells (edge-midpoint rule) and gradients at the centroids."""
    gen = torch.Generator().manual_seed(int(seed))
    x0, x1, y0, y1 = mesh.domain
    P = torch.from_numpy(mesh.xy[mesh.tri]).cuda()
    M = 0.5 * (P + P.roll(-1, 1))
    C = P.mean(1)
    avg, gx, gy = 0, 0, 0
    for _ in range(4):
        a = 2 * float(torch.rand(1, generator=gen)) - 1
        k, ell = (int(torch.randint(1, 4, (1,), generator=gen)) for _ in range(2))
        p, r = (2 * math.pi * float(torch.rand(1, generator=gen)) if periodic else 0.0 for _ in range(2))
        wx, wy = ((2 if periodic else 1) * math.pi * n / w for n, w in ((k, x1 - x0), (ell, y1 - y0)))
        fx, fy = (lambda X: wx * (X[..., 0] - x0) + p), (lambda X: wy * (X[..., 1] - y0) + r)
        avg = avg + a * (torch.cos(fx(M)) * torch.cos(fy(M))).mean(1)
        gx = gx - a * wx * torch.sin(fx(C)) * torch.cos(fy(C))
        gy = gy - a * wy * torch.cos(fx(C)) * torch.sin(fy(C))
    return avg, gx, gy


def _instance_state(problem, mesh, b, seed):
    """Cell averages [6, n] and gradients [6, 2, n] of one instance."""
    dev = torch.device("cuda")
    bm, bg = (torch.from_numpy(v).to(dev) for v in inputs.p1_average_and_gradient(b, mesh))
    P = torch.from_numpy(mesh.xy[mesh.tri]).to(dev)
    x = P[..., 0]
    M = 0.5 * (x + x.roll(-1, 1))
    C = x.mean(1)
    zero = torch.zeros(mesh.n_tri, dtype=torch.float64, device=dev)
    f, fx, fy = _modes(mesh, problem in _PERIODIC, seed)
    amp = {"lake": 1e-3, "circle": 1e-3, "ensemble": 0.02}.get(problem, 0.005)
    top, u = 1.0, (0.0, 0.0)          # free surface and the layers' velocity along x
    if problem == "ridge":
        e, ex = 0.7 - 0.1 * torch.exp(-20 * (M - 1) ** 2).mean(1), 4 * (C - 1) * torch.exp(-20 * (C - 1) ** 2)
    elif problem == "dambreak":
        e, ex = 0.4 + 0.2 * (x < 0).double().mean(1), zero
    elif problem == "circle":
        inside = ((P - 5.0) ** 2).sum(-1) < 4.0
        e, ex, top = 0.2 + 1.6 * inside.double().mean(1), zero, 2.0
    elif problem == "smooth":
        e, ex, top, u = 1.0 + zero, zero, 2.0, (0.1, 0.1)
    elif problem == "lake":
        e, ex = 0.8 + zero, zero
    elif problem == "channel":
        e, ex, top, u = 0.8 + zero, zero, 1.2, (-0.2, 0.15)
    else:
        e, ex = 0.5 + zero, zero
    e, ex, ey = e + amp * f, ex + amp * fx, amp * fy
    avg, grad = torch.zeros(6, mesh.n_tri, dtype=torch.float64, device=dev), torch.zeros(
        6, 2, mesh.n_tri, dtype=torch.float64, device=dev)
    avg[3], grad[3, 0], grad[3, 1] = e - bm, ex - bg[0], ey - bg[1]
    avg[0], grad[0, 0], grad[0, 1] = top - e, -ex, -ey
    for base, vel in ((3, u[0]), (0, u[1])):
        avg[base + 1], grad[base + 1] = vel * avg[base], vel * grad[base]
    return avg, grad


def _state(plan, seed):
    parts = [_instance_state(plan.problem, m, b, 1000 * seed + k) for k, (m, b) in enumerate(zip(plan.meshes, plan.b))]
    return torch.cat([a for a, _ in parts], 1), torch.cat([g for _, g in parts], 2)


def _samples(case, seed):
    """Features, as the gate normalises them, and labels, on the device."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    X = (0.4 * torch.randn(case["n"], 24, generator=gen, device="cuda")).clamp_(-1, 1)
    y = (torch.rand(case["n"], generator=gen, device="cuda") < 0.3).float()
    P = torch.from_numpy(inputs.gate_init(int(seed) % 100003)).cuda()
    P[gks2l.GKS2L_MLP_NTRAIN:gks2l.GKS2L_MLP_NTRAIN + 24] = 0.05 * torch.randn(24, generator=gen, device="cuda")
    P[gks2l.GKS2L_MLP_NTRAIN + 24:] = 1.0 + 0.2 * torch.rand(24, generator=gen, device="cuda")
    return X, y, P


# ----------------------------------------------------------------- interface

def prepare(case, seed):
    if case["kind"] in ("train", "infer"):
        X, y, P = _samples(case, seed)
        s = dict(kind=case["kind"], X=X, y=y, P=P, n=case["n"])
        if case["kind"] == "train":
            z = torch.zeros(gks2l.GKS2L_MLP_NTRAIN, device="cuda")
            s.update(G=z.clone(), m=z.clone(), v=z.clone(), loss=torch.zeros(1, device="cuda"))
        else:
            s["logits"] = torch.empty(case["n"], device="cuda")
        return s
    plan = _plan(case)
    if case["kind"] == "items":
        states = [_state(plan, 64 * seed + i) for i in range(case["items"])]
        pinned = [(a.cpu().pin_memory(), g.cpu().pin_memory()) for a, g in states]
        return dict(kind="items", solver=plan.solver, stages=case["stages"], inputs=pinned,
                    outputs=[(torch.zeros_like(a).pin_memory(), torch.zeros_like(g).pin_memory()) for a, g in pinned])
    avg, grad = _state(plan, seed)
    return dict(kind="flow", solver=plan.solver, fp32=plan.fp32, stages=case["stages"], avg=avg, grad=grad,
                out_avg=torch.empty_like(avg), out_grad=torch.empty_like(grad))


def run(s):
    if s["kind"] == "train":
        gks2l.mlp_grad(s["X"], s["y"], s["P"], 2.0, s["G"], s["loss"])
        gks2l.mlp_adam(s["P"], s["G"], s["m"], s["v"], 1, 3e-3, 1.0 / s["n"])
        return dict(P=s["P"], G=s["G"], m=s["m"], v=s["v"], loss=s["loss"])
    if s["kind"] == "infer":
        gks2l.mlp_forward(s["X"], s["P"], s["logits"])
        return s["logits"]
    if s["kind"] == "items":
        s["solver"].run_items(s["inputs"], s["outputs"], s["stages"])
        return s["outputs"]
    with torch.cuda.stream(s["solver"].stream):
        s["solver"].set_state_device(s["avg"], s["grad"])
        s["solver"].advance(s["stages"], sync=False)
        s["solver"].get_state_device(s["out_avg"], s["out_grad"])
        if s["fp32"]:
            return s["out_avg"].float(), s["out_grad"].float()
    return s["out_avg"], s["out_grad"]


def _cells(case):
    if case["problem"] == "ensemble":
        return int(2 * (inputs.ensemble_sizes(case["instances"], case["lo"], case["hi"]).astype(np.int64) ** 2).sum())
    return 2 * case["nx"] * case["ny"]


def work(case):
    """The method's own counts: the state (18 values a triangle) comes in and
    goes out once, the triangles' 9 x 17 fits are read once, and a stage of one
    triangle takes about 10 kflop (reconstruction 3396, 1.5 edges of
    4096 + 520, update 400)."""
    if case["kind"] in ("train", "infer"):
        passes, out = (3, 4 * (case["n"] + 4 * 1889)) if case["kind"] == "train" else (1, 4 * case["n"])
        return dict(bytes=case["n"] * 96 + out, flops=passes * 2.0 * case["n"] * (24 * 32 + 32 * 32 + 32))
    n, rs = _cells(case), 4 if case["precision"] == "fp32" else 8
    steps = case["stages"] * case.get("items", 1)
    ends = case.get("items", 1) * n * (2 * 18 * 8 + (18 * 4 if rs == 4 else 0))
    return dict(bytes=ends + n * rs * 153, flops=steps * n * 10720.0)


# --------------------------------------------------- the method in 64 bits

def _lookup(key):
    """For each half edge the other one with the same key, or -1."""
    order = np.argsort(key, kind="stable")
    k = key[order]
    same = k[1:] == k[:-1]
    other = np.full(key.size, -1, np.int64)
    other[order[:-1][same]] = order[1:][same]
    other[order[1:][same]] = order[:-1][same]
    return other


def _geometry(mesh, dev):
    """Cells, face images and stencils of a mesh. An image of a cell is (cell,
    A, t): x -> A x + t maps the cell's own frame into the viewer's."""
    tri, xy = mesh.tri.astype(np.int64), mesh.xy
    n = mesh.n_tri
    vid = np.arange(mesh.n_vert)
    if mesh.period[0] > 0:            # one id for all periodic images of a vertex
        i, j = vid % (mesh.nx + 1), vid // (mesh.nx + 1)
        vid = (i % mesh.nx) + mesh.nx * (j % mesh.ny)
    a, b = vid[tri], vid[np.roll(tri, -1, 1)]
    other = _lookup((np.minimum(a, b) * (vid.max() + 1) + np.maximum(a, b)).ravel())
    wall = other < 0
    other[wall] = np.nonzero(wall)[0]
    P = torch.from_numpy(xy[tri]).to(dev)
    other, wall = torch.from_numpy(other).to(dev).view(n, 3), torch.from_numpy(wall).to(dev).view(n, 3)
    d = P.roll(-1, 1) - P
    length = d.norm(dim=-1)
    normal = torch.stack([d[..., 1], -d[..., 0]], -1) / length[..., None]
    mid = 0.5 * (P + P.roll(-1, 1))
    eye = torch.eye(2, dtype=torch.float64, device=dev).expand(n, 3, 2, 2)
    w = wall[..., None]
    A = torch.where(w[..., None], eye - 2 * normal[..., :, None] * normal[..., None, :], eye)
    t = torch.where(w, 2 * (mid * normal).sum(-1, keepdim=True) * normal, mid - mid.view(-1, 2)[other])
    t = torch.where(w | (t.abs() > 1e-9), t, torch.zeros_like(t))
    nb = other // 3
    area = 0.5 * (d[:, 0, 0] * d[:, 1, 1] - d[:, 0, 1] * d[:, 1, 0])
    cen = P.mean(1)
    # stencil: three face images, then the faces of each of them
    cell = torch.cat([nb, nb[nb].view(n, 9)], 1)
    A2 = (A[:, :, None] @ A[nb]).view(n, 9, 2, 2)
    t2 = ((A[:, :, None] @ t[nb][..., None])[..., 0] + t[:, :, None]).view(n, 9, 2)
    SA, St = torch.cat([A, A2], 1), torch.cat([t, t2], 1)
    c = (SA @ cen[cell][..., None])[..., 0] + St
    tol = 1e-6 * area.sqrt()
    near = lambda p, q, cp, cq: ((p - q).abs().amax(-1) <= tol) & (cp == cq)  # noqa: E731
    keep = torch.ones(n, 12, dtype=torch.bool, device=dev)
    own = torch.arange(n, device=dev)
    for s in range(3, 12):
        keep[:, s] = ~near(c[:, s], cen, cell[:, s], own)
        for r in range(s):
            keep[:, s] &= ~(keep[:, r] & near(c[:, s], c[:, r], cell[:, s], cell[:, r]))
    return dict(n=n, P=P, other=other, wall=wall, length=length, normal=normal, mid=mid, A=A, nb=nb, area=area,
                cen=cen, hs=area.sqrt(), cell=cell, SA=SA, St=St, keep=keep, dX=4 * area / length.sum(1))


def _rule(m):
    x, w = np.polynomial.legendre.leggauss(m)
    x, w = 0.5 * (x + 1), 0.5 * w
    a, b = np.meshgrid(x, x, indexing="ij")
    v = np.outer(w, w) * (1 - a)
    return a.ravel(), (b * (1 - a)).ravel(), (v / v.sum()).ravel()


def _monomials(x, y):
    """Taylor monomials of degree 1..3 and their x- and y-derivatives."""
    o, z = torch.ones_like(x), torch.zeros_like(x)
    m = (x, y, x * x / 2, x * y, y * y / 2, x ** 3 / 6, x * x * y / 2, x * y * y / 2, y ** 3 / 6)
    mx = (o, z, x, y, z, x * x / 2, x * y, y * y / 2, z)
    my = (z, o, z, x, y, z, x * x / 2, x * y, y * y / 2)
    return torch.stack(m, -1), torch.stack(mx, -1), torch.stack(my, -1)


def _pinv(A):
    """Pseudo-inverse of full-rank columns, by Gram-Schmidt done twice."""
    k = A.shape[-1]
    Q, R = A.clone(), torch.zeros(A.shape[0], k, k, dtype=A.dtype, device=A.device)
    for j in range(k):
        for _ in range(2):
            if j:
                s = (Q[..., :j] * Q[..., j:j + 1]).sum(1)
                Q[..., j] -= (Q[..., :j] * s[:, None, :]).sum(-1)
                R[:, :j, j] += s
        R[:, j, j] = Q[..., j].norm(dim=1)
        Q[..., j] /= R[:, j, j, None]
    out = Q.transpose(1, 2).clone()
    for i in range(k - 1, -1, -1):
        for j in range(i + 1, k):
            out[:, i] -= R[:, i, j, None] * out[:, j]
        out[:, i] /= R[:, i, i, None]
    return out


def _operators(G):
    n, hs, cen = G["n"], G["hs"], G["cen"]
    qa, qb, qw = (torch.from_numpy(v).to(hs.device) for v in _rule(4))

    def average(T):
        """Cell averages over triangles T of the scaled monomials and their derivatives."""
        X = T[:, 0, None] + qa[:, None] * (T[:, 1] - T[:, 0])[:, None] + qb[:, None] * (T[:, 2] - T[:, 0])[:, None]
        X = (X - cen[:, None]) / hs[:, None, None]
        return [(v * qw[:, None]).sum(1) for v in _monomials(X[..., 0], X[..., 1])]

    image = lambda s: (G["SA"][:, s, None] @ G["P"][G["cell"][:, s]][..., None])[..., 0] + G["St"][:, s, None]  # noqa: E731
    m0, mx, my = average(G["P"])
    rows, grads = [], [mx, my]
    for s in range(12):
        im, ix, iy = average(image(s))
        rows.append((im - m0) * G["keep"][:, s, None])
        if s < 3:
            grads += [ix, iy]
    lsq = _pinv(torch.stack(rows + grads, 1))                       # [n, 9, 12 + 8]
    p1 = []
    for f in range(3):
        B = torch.stack([rows[f][:, :2]] + [g[:, :2] for g in (mx, my, grads[2 + 2 * f], grads[3 + 2 * f])], 1)
        p1.append(_pinv(B))
    # smoothness form: mean of the squared derivatives of order 1 and 2, plus the third ones
    X = G["P"][:, 0, None] + qa[:, None] * (G["P"][:, 1] - G["P"][:, 0])[:, None] + \
        qb[:, None] * (G["P"][:, 2] - G["P"][:, 0])[:, None]
    X = (X - cen[:, None]) / hs[:, None, None]
    x, y = X[..., 0], X[..., 1]
    _, dx, dy = _monomials(x, y)
    o, z = torch.ones_like(x), torch.zeros_like(x)
    second = [torch.stack(v, -1) for v in ((z, z, o, z, z, x, y, z, z), (z, z, z, o, z, z, x, y, z),
                                           (z, z, z, z, o, z, z, x, y))]
    form = sum(torch.einsum("q,nqa,nqb->nab", qw, v, v) for v in [dx, dy] + second)
    form[:, range(5, 9), range(5, 9)] += 1.0
    # the plane through the three edge midpoints
    M = G["mid"]
    plane = torch.linalg.inv(torch.stack([M[:, 1] - M[:, 0], M[:, 2] - M[:, 0]], 1))
    # Gauss points of each face, and the monomials there
    g = 0.5 / math.sqrt(3.0)
    d = G["P"].roll(-1, 1) - G["P"]
    X = (M[:, :, None] + torch.tensor([-g, g], dtype=torch.float64, device=hs.device)[:, None] * d[:, :, None])
    S = (X - cen[:, None, None]) / hs[:, None, None, None]
    pm, px, py = _monomials(S[..., 0], S[..., 1])                   # [n, 3, 2, 9]
    return dict(lsq=lsq, p1=p1, form=form, plane=plane, m0=m0, pm=pm - m0[:, None, None], px=px, py=py)


def _vectors(A, x, y):
    return A[..., 0, 0] * x + A[..., 0, 1] * y, A[..., 1, 0] * x + A[..., 1, 1] * y


def _image_values(A, avg, grad, cells):
    """Averages [6] and gradients [6][2] of cells seen through A."""
    q = [avg[v][cells] for v in range(6)]
    g = [[grad[v, 0][cells], grad[v, 1][cells]] for v in range(6)]
    for b in (1, 4):
        q[b], q[b + 1] = _vectors(A, q[b], q[b + 1])
        T = [_vectors(A, g[b][k], g[b + 1][k]) for k in range(2)]   # rotate the components, then the directions
        g[b], g[b + 1] = [_vectors(A, T[0][i], T[1][i]) for i in range(2)]
    for v in (0, 3):
        g[v] = _vectors(A, *g[v])
    return q, g


def _reconstruct(G, O, Q, D, smooth, par):
    """Coefficients [6][n, 9] about the averages, and omega_H / gamma_H [6][n].
    Q, D: averages and gradients with variable 3 as the water level."""
    hs, gh = G["hs"], 0.85
    gl = (1 - gh) / 3
    q, _ = _image_values(G["SA"], Q, D, G["cell"])
    _, g = _image_values(G["A"], Q, D, G["nb"])
    coef, fac = [], []
    for v in range(6):
        rhs = [torch.where(G["keep"], q[v] - Q[v][:, None], 0.0), hs[:, None] * D[v].T]
        rhs.append((hs[:, None, None] * torch.stack(list(g[v]), -1)).view(-1, 6))
        r = torch.cat(rhs, 1)
        a = (O["lsq"] @ r[..., None])[..., 0]
        b = [(O["p1"][f] @ torch.stack([r[:, f], r[:, 12], r[:, 13], r[:, 14 + 2 * f], r[:, 15 + 2 * f]], 1)[..., None])
             [..., 0] for f in range(3)]
        beta = [torch.einsum("na,nab,nb->n", a, O["form"], a)] + [(x * x).sum(1) for x in b]
        tz = sum((beta[0] - x).abs() for x in beta[1:]) / 3
        eps = G["area"] * (1 + Q[v] ** 2)
        w = [gm * (1 + (tz / (x + eps)) ** 2) for gm, x in zip((gh, gl, gl, gl), beta)]
        total = sum(w)
        w = [x / total for x in w]
        if smooth is not None:
            w = [torch.where(smooth, gm, x) for gm, x in zip((gh, gl, gl, gl), w)]
        f0 = w[0] / gh
        c = f0[:, None] * a
        c[:, :2] += sum((w[1 + k] - f0 * gl)[:, None] * b[k] for k in range(3))
        coef.append(c)
        fac.append(f0)
    return coef, fac


def _half_moments(U, th, sign):
    """Central moments 0..5 of the unit Maxwellian over sign * u > 0."""
    E = sign * torch.exp(-U * U / (2 * th)) * torch.sqrt(th / (2 * math.pi))
    mu = [0.5 * (1 + sign * torch.erf(U / torch.sqrt(2 * th))), E]
    for k in range(1, 5):
        mu.append(k * th * mu[k - 1] + (-U) ** k * E)
    return mu


def _slopes(h, U, V, th, dn, dt, F):
    """Slope and force of a Maxwellian as a polynomial in c = u - U: the terms
    {(power of cu, power of cv): coefficient}."""
    lam = 0.5 / th
    un, vn = (dn[1] - U * dn[0]) / h, (dn[2] - V * dn[0]) / h
    ut, vt = (dt[1] - U * dt[0]) / h, (dt[2] - V * dt[0]) / h
    al = lam * (U * dn[0] + V * dt[0]) / h
    fu, fv = lam * F[0] / h, lam * F[1] / h
    return {(1, 0): 2 * lam * (un * U + ut * V), (0, 1): 2 * lam * (vn * U + vt * V), (2, 0): al + 2 * lam * un,
            (0, 2): al + 2 * lam * vt, (1, 1): 2 * lam * (vn + ut), (3, 0): fu, (1, 2): fu, (2, 1): fv, (0, 3): fv}


def _moments(K, mu, th, U, V):
    """Moments of K with 1, u, v and u, u u, u v."""
    nv = {0: 1.0, 2: th, 4: 3 * th * th}

    def m(i, j):
        return sum(c * mu[a + i] * nv[b + j] for (a, b), c in K.items() if (b + j) % 2 == 0)
    t00, t10, t20, t01, t11 = m(0, 0), m(1, 0), m(2, 0), m(0, 1), m(1, 1)
    o1 = U * t00 + t10
    return [t00, o1, V * t00 + t01, o1, U * U * t00 + 2 * U * t10 + t20, U * V * t00 + V * t10 + U * t01 + t11]


def _interface(l, r, g, tau, dt):
    """Flux and interface variables at a stage start and their time
    derivatives, in the face's frame. l, r: (h, U, V, dn, dt, F)."""
    sides = []
    for (h, U, V, dn, dtt, F), sign in ((l, 1.0), (r, -1.0)):
        th = 0.5 * g * h
        sides.append((h, U, V, th, _half_moments(U, th, sign), _slopes(h, U, V, th, dn, dtt, F)))
    c1 = [lambda mu, U, V, th: mu[0], lambda mu, U, V, th: U * mu[0] + mu[1], lambda mu, U, V, th: V * mu[0],
          lambda mu, U, V, th: U * mu[0] + mu[1], lambda mu, U, V, th: U * U * mu[0] + 2 * U * mu[1] + mu[2],
          lambda mu, U, V, th: V * (U * mu[0] + mu[1])]
    p3 = [sum(h * f(mu, U, V, th) for h, U, V, th, mu, _ in sides) for f in c1]
    h, U, V = p3[0], p3[1] / p3[0], p3[2] / p3[0]
    th = 0.5 * g * h
    p0 = [h, h * U, h * V, h * U, h * U * U + th * h, h * U * V]
    p1 = 0
    for (_, _, _, dn, dtt, F), sign in ((l, 1.0), (r, -1.0)):
        m = _moments(_slopes(h, U, V, th, dn, dtt, F), _half_moments(U, th, sign), th, U, V)
        p1 = [h * x for x in m] if p1 == 0 else [p + h * x for p, x in zip(p1, m)]
    d = [-p1[0], -p1[1], -p1[2]]
    p2 = d + [d[1], 2 * U * d[1] - U * U * d[0] + 2 * th * d[0], V * d[1] + U * d[2] - U * V * d[0]]
    p4 = 0
    for hh, UU, VV, tt, mu, K in sides:
        m = _moments(K, mu, tt, UU, VV)
        p4 = [hh * x for x in m] if p4 == 0 else [p + hh * x for p, x in zip(p4, m)]

    def integrals(x):
        e, em = torch.exp(-x / tau), -torch.expm1(-x / tau)
        return (x - tau * em, -tau * x * (1 + e) + 2 * tau ** 2 * em, x * x / 2 - tau * x + tau ** 2 * em, tau * em,
                tau * x * e - tau ** 2 * em)
    full, half = integrals(dt), integrals(dt / 2)
    value = [(4 * b - a) / dt for a, b in zip(full, half)]
    rate = [4 * (a - 2 * b) / dt ** 2 for a, b in zip(full, half)]
    at = lambda w, k: sum(c * p[k] for c, p in zip(w, (p0, p1, p2, p3, p4)))  # noqa: E731
    return [[at(w, k + s) for k in range(3)] for s, w in ((3, value), (3, rate), (0, value), (0, rate))]


def _features(G, Q, D):
    """The gate's 24 inputs."""
    _, g = _image_values(G["A"], Q, D, G["nb"])
    out = []
    for v in (3, 0):
        q = torch.cat([Q[v][:, None], Q[v][G["nb"]]], 1)
        dev = q - q.mean(1, keepdim=True)
        raw = [torch.stack([dev[:, 0], G["hs"] * D[v, 0], G["hs"] * D[v, 1]], 1)]
        raw += [torch.stack([dev[:, 1 + f], G["hs"] * g[v][0][:, f], G["hs"] * g[v][1][:, f]], 1) for f in range(3)]
        raw = torch.cat(raw, 1)
        out.append(raw / torch.sqrt((raw ** 2).sum(1) + G["area"] * (1 + Q[v] ** 2))[:, None])
    return torch.cat(out, 1)


def _logits(P, X):
    P = P.double()
    w1, b1, w2, b2 = P[:768].view(32, 24), P[768:800], P[800:1824].view(32, 32), P[1824:1856]
    x = (X.double() - P[1889:1913]) * P[1913:]
    return torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2) @ P[1856:1888] + P[1888]


class _Exact:
    """The two-layer scheme on one mesh in plain double precision."""

    def __init__(self, mesh, b, avg, grad, chi, floor, network):
        dev = avg.device
        self.G = _geometry(mesh, dev)
        self.O = _operators(self.G)
        bm, bg = (torch.from_numpy(v).to(dev) for v in inputs.p1_average_and_gradient(b, mesh))
        G = self.G
        self.bm, self.bg, self.g, self.chi, self.floor, self.network = bm, bg, 9.81, chi, floor, network
        # the bottom is continuous and linear in each cell: its values at the Gauss points
        bp = _gauss_points(G)
        self.bq = bm[:, None, None] + ((bp - G["cen"][:, None, None]) * bg.T[:, None, None]).sum(-1)
        self.avg, self.grad = avg.clone(), grad.clone()
        self.smooth = self.gate()

    def levels(self):
        Q, D = self.avg.clone(), self.grad.clone()
        Q[3] += self.bm
        D[3] += self.bg
        return Q, D

    def gate(self):
        if self.network is None:
            return None
        return _logits(self.network, _features(self.G, *self.levels())) < math.log(gate.THRESHOLD / (1 - gate.THRESHOLD))

    def opposite(self, x):
        """The neighbour's values at the same Gauss points (its points run the
        other way); a wall's neighbour is the cell itself, its points its own."""
        G = self.G
        y = x.reshape(3 * G["n"], 2)[G["other"].reshape(-1)].view(G["n"], 3, 2)
        return torch.where(G["wall"][..., None], y, y.flip(-1))

    def stage(self, stage, dt):
        G, O, g = self.G, self.O, self.g
        Q, D = self.levels()
        coef, fac = _reconstruct(G, O, Q, D, self.smooth, None)
        following = self.gate()
        ev = lambda c, m: torch.einsum("nk,nfqk->nfq", c, m)  # noqa: E731
        depth_bar, flagged = [self.avg[3], self.avg[0]], [None, None]
        if self.floor:
            for lay, base in ((0, 3), (1, 0)):
                h = Q[base][:, None, None] + ev(coef[base], O["pm"]) - (self.bq if lay == 0 else 0)
                low, bar = h.amin((1, 2)), depth_bar[lay]
                flagged[lay] = low < 0.5 * bar
                th = torch.where(low < self.floor * bar, (bar - self.floor * bar) / (bar - low), 1.0).clamp(min=0.0)
                for v in range(base, base + 3):
                    coef[v] = coef[v] * th[:, None]
                if lay == 0:
                    coef[3][:, :2] += ((1 - th) * G["hs"] * self.bg).T
        val = [Q[v][:, None, None] + ev(coef[v], O["pm"]) for v in range(6)]
        slope = [[ev(coef[v], O[d]) / G["hs"][:, None, None] for d in ("px", "py")] for v in range(6)]
        A = G["A"][:, :, None]
        other = [self.opposite(x) for x in val]
        oslope = [[self.opposite(x) for x in s] for s in slope]
        for b in (1, 4):
            other[b], other[b + 1] = _vectors(A, other[b], other[b + 1])
            T = [_vectors(A, oslope[b][k], oslope[b + 1][k]) for k in range(2)]
            oslope[b], oslope[b + 1] = [list(_vectors(A, T[0][i], T[1][i])) for i in range(2)]
        for v in (0, 3):
            oslope[v] = list(_vectors(A, *oslope[v]))
        obg = _vectors(G["A"], self.bg[0][G["nb"]], self.bg[1][G["nb"]])
        nx, ny = G["normal"][..., 0, None], G["normal"][..., 1, None]
        nt = lambda x, y: (x * nx + y * ny, y * nx - x * ny)  # noqa: E731
        # blended levels and their planes
        blend, plane, oplane = {}, {}, {}
        for base in (3, 0):
            bot = self.bq if base == 3 else 0
            hl, hr = val[base] - bot, other[base] - bot
            ul, ur = nt(val[base + 1], val[base + 2])[0] / hl, nt(other[base + 1], other[base + 2])[0] / hr
            xi = 0.5 * torch.erfc(0.5 * (ul + ur))
            c = (other[base] + xi * (val[base] - other[base])).mean(-1)
            blend[base] = c
            pg = (O["plane"] @ torch.stack([c[:, 1] - c[:, 0], c[:, 2] - c[:, 0]], 1)[..., None])[..., 0]
            plane[base] = (pg[:, 0, None, None], pg[:, 1, None, None])
            oplane[base] = [x[..., None] for x in _vectors(G["A"], pg[:, 0][G["nb"]], pg[:, 1][G["nb"]])]
        flux, rate, W, Wt = ([None] * 6 for _ in range(4))
        for base in (3, 0):
            oth, cf, lay = 3 - base, self.chi if base == 3 else 1.0, 0 if base == 3 else 1
            w = torch.minimum(fac[oth][:, None], fac[oth][G["nb"]]).clamp(0, 1)[..., None]
            bot = self.bq if base == 3 else 0
            pair = []
            for V, S, B, pl in ((val, slope, self.bg, plane), (other, oslope, obg, oplane)):
                h = V[base] - bot
                un, ut = nt(V[base + 1] / h, V[base + 2] / h)
                if base != 3:
                    gb = (0.0, 0.0)
                elif V is val:
                    gb = (B[0][:, None, None], B[1][:, None, None])
                else:
                    gb = (B[0][..., None], B[1][..., None])
                dh = nt(S[base][0] - gb[0], S[base][1] - gb[1])
                mx, my = nt(*S[base + 1]), nt(*S[base + 2])
                F = nt(*(S[base][k] + cf * (w * S[oth][k] + (1 - w) * pl[oth][k]) for k in range(2)))
                dirs = [(dh[k],) + nt(mx[k], my[k]) for k in range(2)]
                pair.append([h, un, ut, dirs[0], dirs[1], F])
            if self.floor:
                bar = depth_bar[lay]
                mean = [[x[..., None].expand_as(val[0]) for x in (y[:, None].expand(-1, 3) for y in
                        (self.avg[base + 1] / bar, self.avg[base + 2] / bar))]]
                mean.append([x[..., None].expand_as(val[0]) for x in
                             _vectors(G["A"], *((self.avg[base + k] / bar)[G["nb"]] for k in (1, 2)))])
                un, ut = zip(*(nt(*x) for x in mean))
                fl = [flagged[lay][:, None, None], flagged[lay][G["nb"]][..., None]]
                for sd in range(2):
                    for k, u in ((1, un), (2, ut)):
                        inside = torch.maximum(torch.minimum(pair[sd][k], torch.maximum(*u)), torch.minimum(*u))
                        pair[sd][k] = torch.where(fl[sd], inside, pair[sd][k])
            hl, hr = pair[0][0], pair[1][0]
            tau = (0.05 + 5.0 * ((hl * hl - hr * hr) / (hl * hl + hr * hr)).abs()) * dt
            for out, x in zip((flux, rate, W, Wt), _interface(*pair, g, tau, dt)):
                out[base] = x[0].mean(-1)
                out[base + 1] = (x[1] * nx - x[2] * ny).mean(-1)
                out[base + 2] = (x[1] * ny + x[2] * nx).mean(-1)
            W[base] = W[base] + (self.bq.mean(-1) if base == 3 else 0)      # the water level
        s = G["length"] / G["area"][:, None]
        gauss = lambda x: torch.stack([(s * G["normal"][..., k] * x).sum(1) for k in range(2)])  # noqa: E731
        L, Lt = ([-(s * x).sum(1) for x in v] for v in (flux, rate))
        if stage == 1:
            self.W0 = W
        end = [self.W0[v] + (0.5 if stage == 1 else 1.0) * dt * Wt[v] for v in range(6)]
        own = {b: val[b].mean(-1) for b in (3, 0)}
        m2, m1 = own[0].mean(1), own[3].mean(1) - self.bm
        t2, t1 = Wt[0].mean(1), Wt[3].mean(1)
        d1, d2 = gauss(own[3]) - self.bg, gauss(own[0])
        for k in range(2):
            L[1 + k] = L[1 + k] - g * self.avg[0] * self.bg[k] - g * m2 * d1[k]
            Lt[1 + k] = Lt[1 + k] - g * L[0] * self.bg[k] - g * (t2 * d1[k] + m2 * gauss(Wt[3])[k])
            L[4 + k] = L[4 + k] - g * self.avg[3] * self.bg[k] - self.chi * g * m1 * d2[k]
            Lt[4 + k] = Lt[4 + k] - g * L[3] * self.bg[k] - self.chi * g * (t1 * d2[k] + m1 * gauss(Wt[0])[k])
        L, Lt = torch.stack(L), torch.stack(Lt)
        if stage == 1:
            self.start = (self.avg, L, Lt)
            self.avg = self.avg + dt / 2 * L + dt * dt / 8 * Lt
        else:
            a, L0, Lt0 = self.start
            self.avg = a + dt * L0 + dt * dt / 6 * Lt0 + dt * dt / 3 * Lt
        self.grad = torch.stack([gauss(x) for x in end])
        self.grad[3] -= self.bg
        self.smooth = following

    def advance(self, stages):
        for k in range(stages):
            if k % 2 == 0:
                speed = [((self.avg[b + 1] ** 2 + self.avg[b + 2] ** 2).sqrt() / self.avg[b] +
                          (self.g * self.avg[b]).sqrt()) for b in (0, 3)]
                self.dt = 0.5 * (self.G["dX"] / torch.maximum(*speed)).min()
            self.stage(1 + k % 2, self.dt)
        return self.avg, self.grad


def _gauss_points(G):
    """The faces' Gauss points [n, 3, 2, 2]."""
    g = torch.tensor([-0.5, 0.5], dtype=torch.float64, device=G["P"].device) / math.sqrt(3.0)
    return G["mid"][:, :, None] + g[:, None] * (G["P"].roll(-1, 1) - G["P"])[:, :, None]


def _exact_flow(problem, meshes, bs, states, stages, floor, network):
    parts = [_Exact(m, b, a, g, _CHI.get(problem, 0.98), floor, network).advance(stages)
             for m, b, (a, g) in zip(meshes, bs, states)]
    return torch.cat([a for a, _ in parts], 1), torch.cat([g for _, g in parts], 2)


def exact(case, seed):
    if case["kind"] == "infer":
        X, _, P = _samples(case, seed)
        return _logits(P, X)
    if case["kind"] == "train":
        X, y, P = _samples(case, seed)
        P = P.double().requires_grad_()
        s = _logits(P, X)
        loss = (2.0 * y * torch.nn.functional.softplus(-s) + (1 - y) * torch.nn.functional.softplus(s)).sum()
        G = torch.autograd.grad(loss, P)[0][:gks2l.GKS2L_MLP_NTRAIN]
        r = G / case["n"]
        new = P.detach().clone()
        new[:r.numel()] -= 3e-3 * r / (r.abs() + 1e-8)             # Adam's first step
        return dict(P=new, G=G, m=0.1 * r, v=0.001 * r * r, loss=loss.detach().view(1))
    plan = _plan(case)
    network = torch.from_numpy(_network()).cuda() if case.get("gate") else None

    def flow(k):
        states = [_instance_state(plan.problem, m, b, 1000 * k + i)
                  for i, (m, b) in enumerate(zip(plan.meshes, plan.b))]
        return _exact_flow(plan.problem, plan.meshes, plan.b, states, case["stages"], case.get("positivity", 0.0),
                           network)
    if case["kind"] == "items":
        return [flow(64 * seed + i) for i in range(case["items"])]
    return flow(seed)
