"""Workloads by which the speed of this framework is measured.

Each case is one call sequence of a user's program through the public entry
points, over the sizes of the repository's configurations and tests:

  run      a notched plate or a fragmentation plate resumed from a saved state
           and stepped while it cracks (the checkpoint/restart of long runs and
           of parameter studies; every pass does the same steps)
  elastic  a large plate stepped before its first split (wave propagation and
           the evaluation of every surface point), the fields read on the device
  batch    a specimen sweep: many plates resumed and stepped in one batch
  tri      an unstructured triangle mesh stepped, the fields read on the device
  layer    one 3x3 convolution layer of the surrogate: forward with bias and
           ReLU, data gradient with the ReLU mask, weight and bias gradients
  infer    the surrogate's forward pass
  grads    the surrogate's training pass: forward, loss, every gradient

A case names its family in "kind".  `exact` gives the 64-bit result of the
elastic, triangle, layer and surrogate families (of the training pass, its
logits and loss); a cracking run has none here (which element splits next
hangs on the last bits).
"""
import ctypes
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_2509_01827_gb300 import cem, inputs, surrogate

FP64, FP32 = cem.CEM_FP64, cem.CEM_FP32_MIXED
DEV = "cuda:0"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest configuration whole: 4,000 elements, 2000 FP64 steps,
        # latency- and launch-bound
        dict(name="notched_100x40_fp64", kind="run", plate="notched", nx=100, ny=40,
             precision=FP64, begin=1, steps=2000),
        # the branching plate at 0.25 mm to 80 us, as the surrogate's data set
        # and the crack studies run it
        dict(name="notched_400x160_fp32", kind="run", plate="notched", nx=400, ny=160,
             precision=FP32, begin=1, steps=2440),
        # the same plate in the reference precision
        dict(name="notched_400x160_fp64", kind="run", plate="notched", nx=400, ny=160,
             precision=FP64, begin=1, steps=2440),
        # a fragmenting plate with many tips at once, resumed past initiation
        dict(name="fragmentation_1024_fp32", kind="run", plate="fragmentation", nx=1024, ny=1024,
             precision=FP32, begin=250, steps=600),
        # the flagship mesh, 4.2 M elements, before its first split
        dict(name="elastic_2048_fp32", kind="elastic", n=2048, precision=FP32, steps=64),
        dict(name="elastic_2048_fp64", kind="elastic", n=2048, precision=FP64, steps=8),
        # the specimen sweep: 64 plates of 100x40 .. 400x160
        dict(name="specimens_64_fp32", kind="batch", count=64, smin=1.0, smax=4.0,
             precision=FP32, begin=100, steps=500),
        # a million triangles
        dict(name="tri_1024x512_fp32", kind="tri", nx=1024, ny=512, precision=FP32, steps=64),
        # a full-resolution layer of the surrogate at the training batch: few
        # channels, many pixels
        dict(name="layer_full_32", kind="layer", B=64, H=160, W=400, cin=32, cout=32, pad=0),
        # the bottom layer: many channels, few pixels
        dict(name="layer_deep_512", kind="layer", B=64, H=10, W=25, cin=512, cout=512, pad=0),
        # one image through the network
        dict(name="infer_b1", kind="infer", B=1, H=160, W=400, levels=5),
        # a training pass of the batch the trainer uses
        dict(name="grads_b64", kind="grads", B=64, H=160, W=400, levels=5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "elastic", "batch", "tri", "layer", "layer", "infer", "grads"])
    prec = rng.choice([FP32, FP64])
    if kind == "run":
        if rng.random() < 0.5:
            nx = _log(rng, 40, 400)
            ny = max(16, int(nx * rng.uniform(0.3, 0.6)))
            return dict(kind=kind, plate="notched", nx=nx, ny=ny, precision=prec,
                        begin=rng.randint(1, 50), steps=_log(rng, 200, 2000))
        n = _log(rng, 64, 1024 if prec == FP32 else 384)
        return dict(kind=kind, plate="fragmentation", nx=n, ny=n, precision=prec,
                    begin=max(1, int(rng.uniform(0.8, 1.1) * 250 * n / 1024)),
                    steps=_log(rng, 50, 400))
    if kind == "elastic":
        n = _log(rng, 64, 2000 if prec == FP32 else 1400)
        return dict(kind=kind, n=n, precision=prec, steps=_log(rng, 1, 64 if prec == FP32 else 16))
    if kind == "batch":
        a = rng.uniform(0.5, 2.0)
        return dict(kind=kind, count=_log(rng, 2, 64), smin=a, smax=a * rng.uniform(1.1, 2.0),
                    precision=prec, begin=rng.randint(1, 100), steps=_log(rng, 50, 400))
    if kind == "tri":
        return dict(kind=kind, nx=_log(rng, 30, 700), ny=_log(rng, 30, 500), precision=prec,
                    steps=_log(rng, 1, 64))
    if kind == "layer":
        # image sizes of every level and odd ones, channel counts in eights
        H, W = _log(rng, 5, 160), _log(rng, 5, 400)
        cin, cout = 8 * _log(rng, 1, 96), 8 * _log(rng, 1, 64)
        most = 1.5e11 / (2 * 9 * H * W * cin * cout)
        B = _log(rng, 1, max(1, min(64, int(most))))
        return dict(kind=kind, B=B, H=H, W=W, cin=cin, cout=cout, pad=rng.choice([0, 0, 8, 32]))
    levels = rng.randint(2, 5)
    m = 1 << (levels - 1)
    H, W = m * max(1, _log(rng, 16, 160) // m), m * max(1, _log(rng, 24, 400) // m)
    return dict(kind=kind, B=_log(rng, 1, 64 if kind == "infer" else 32), H=H, W=W, levels=levels)


# -------------------------------------------------------------- the plates
def _notched(case, seed):
    """The notched plate with a seeded traction and Weibull G_c field."""
    r = np.random.default_rng([seed, 1])
    p = inputs.notched_plate(case["nx"], case["ny"], traction=1e6 * r.uniform(0.9, 1.1),
                             phantom_cap=max(8192, 4 * case["nx"] * case["ny"]),
                             crack_cap=max(4096, case["nx"] * case["ny"]))
    return dataclasses.replace(p, gc=_weibull(r, p.n_elems))


def _weibull(r, n):
    lam = 3.0 / math.gamma(1.1)
    return (lam * r.weibull(10.0, n)).astype(np.float32)


@functools.lru_cache(maxsize=4)
def _plate(n, p0):
    # the mesh, its hole and rim; the G_c field follows per seed
    return inputs.fragmentation(n, p0=p0, phantom_cap=max(8192, n * n // 4),
                                crack_cap=max(8192, n * n // 8))


def _fragmentation(n, seed, p0):
    r = np.random.default_rng([seed, 2])
    p = _plate(n, p0)
    return dataclasses.replace(p, gc=_weibull(r, p.n_elems))


def _modes(nx, ny, hx, hy, seed):
    """A seeded smooth velocity field of a few cm/s (far below cracking)."""
    r = np.random.default_rng([seed, 3])
    x = np.arange(nx + 1) / nx
    y = np.arange(ny + 1)[:, None] / ny
    v = []
    for _ in range(2):
        f = np.zeros((ny + 1, nx + 1))
        for _ in range(3):
            kx, ky, a, b = r.integers(1, 9), r.integers(1, 9), r.uniform(0, 6.28), r.uniform(0, 6.28)
            f += np.sin(2 * np.pi * kx * x + a) * np.sin(2 * np.pi * ky * y + b)
        v.append(0.02 * f.reshape(-1))
    return v


def _fields(s, n):
    """Displacement and velocity of the n nodes, FP64 on the device."""
    out = []
    for which in (cem.CEM_FIELD_U, cem.CEM_FIELD_V):
        f = torch.empty(2 * n, dtype=torch.float64, device=DEV)
        rc = cem.lib().cem_get_fields(s.h, which, f.data_ptr(), 16 * n, 1)
        if rc != cem.CEM_OK:
            raise cem.CemError(rc, cem.cem_last_error(s.h))
        out.append(f)
    return out


# ---------------------------------------------------------------- prepare
def prepare(case, seed):
    return {"run": _prep_run, "elastic": _prep_elastic, "batch": _prep_batch, "tri": _prep_tri,
            "layer": _prep_layer, "infer": _prep_net, "grads": _prep_net}[case["kind"]](case, seed)


def _prep_run(case, seed):
    if case["plate"] == "notched":
        p = _notched(case, seed)
    else:
        p = _fragmentation(case["nx"], seed, 50e6)
    s = cem.Solver(p, precision=case["precision"])
    s.step(case["begin"])
    return {"case": case, "solver": s, "blob": s.save_state()}


def _elastic_problem(case, seed):
    return _fragmentation(case["n"], seed, 2e6)


def _prep_elastic(case, seed):
    p = _elastic_problem(case, seed)
    s = cem.Solver(p, precision=case["precision"])
    vx, vy = _modes(p.nx, p.ny, p.hx, p.hy, seed)
    s.set_state(vx=vx, vy=vy)
    return {"case": case, "solver": s, "n": p.n_nodes}


def _prep_batch(case, seed):
    # the sweep's sizes, notches and tractions, with a seeded G_c field each
    probs = inputs.batch_specimens(case["count"], smin=case["smin"], smax=case["smax"])
    r = np.random.default_rng([seed, 5])
    probs = [dataclasses.replace(p, gc=_weibull(r, p.n_elems)) for p in probs]
    members = [cem.Solver(p, precision=case["precision"]) for p in probs]
    b = cem.Batch(members)
    b.step(case["begin"])
    b.close()
    return {"case": case, "members": members, "blobs": [m.save_state() for m in members],
            "n": [p.n_nodes for p in probs]}


@functools.lru_cache(maxsize=2)
def _tri_mesh(nx, ny):
    return inputs.tri_plate(nx, ny, lx=0.1, ly=0.1 * ny / nx, traction=1e6)


def _tri_problem(case, seed):
    p = _tri_mesh(case["nx"], case["ny"])
    r = np.random.default_rng([seed, 4])
    h = 0.1 / case["nx"]
    nn = p.n_nodes
    init = (1e-4 * h * r.standard_normal(nn), 1e-4 * h * r.standard_normal(nn),
            0.1 * r.standard_normal(nn), 0.1 * r.standard_normal(nn))
    return dataclasses.replace(p, init=init)


def _prep_tri(case, seed):
    p = _tri_problem(case, seed)
    return {"case": case, "solver": cem.TriSolver(p, precision=case["precision"]), "n": p.n_nodes}


def _layer_tensors(case, seed):
    """x: a ReLU output; dy: a masked output gradient; FP32 weights and bias."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    B, H, W, cin, cout = (case[k] for k in ("B", "H", "W", "cin", "cout"))
    P = B * H * W
    x = torch.randn(P, cin, device=DEV, generator=g).clamp_(min=0).to(torch.bfloat16)
    dy = 1e-3 * torch.randn(P, cout, device=DEV, generator=g)
    dy = (dy * (torch.rand(P, cout, device=DEV, generator=g) < 0.5)).to(torch.bfloat16)
    w = torch.randn(cout, 3, 3, cin, device=DEV, generator=g) * math.sqrt(2.0 / (9 * cin))
    b = 0.1 * torch.randn(cout, device=DEV, generator=g)
    return x, dy, w.to(torch.bfloat16), b


def _prep_layer(case, seed):
    x, dy, w, b = _layer_tensors(case, seed)
    B, H, W, cin, cout, pad = (case[k] for k in ("B", "H", "W", "cin", "cout", "pad"))
    P = B * H * W
    # the data gradient's transposed, flipped weights, and the output as a
    # channel slice of a wider tensor when pad > 0 (concatenation)
    wt = w.flip(1, 2).permute(3, 1, 2, 0).contiguous()
    ws_bytes = surrogate.sg().cem_sg_wgrad_workspace(B, H, W, cin, cout)
    return dict(case=case, x=x, dy=dy, w=w, wt=wt, b=b,
                y=torch.zeros(P, pad + cout, dtype=torch.bfloat16, device=DEV),
                dx=torch.empty(P, cin, dtype=torch.bfloat16, device=DEV),
                dw=torch.empty(cout, 3, 3, cin, device=DEV), db=torch.empty(cout, device=DEV),
                ws=torch.empty(ws_bytes, dtype=torch.uint8, device=DEV), ws_bytes=ws_bytes)


def _chans(case):
    return [32 << l for l in range(case["levels"])]


def _net_inputs(case, seed):
    """Images as the trainer encodes them (traction, notch, normalised G_c,
    five zero channels) and targets with 7% cracked elements."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    B, P = case["B"], case["H"] * case["W"]
    x = torch.zeros(B, P, 8, device=DEV)
    x[..., 0] = (0.5 + 2.5 * torch.rand(B, 1, device=DEV, generator=g)) / 3
    x[..., 1] = (torch.rand(B, P, device=DEV, generator=g) < 0.01).float()
    x[..., 2] = torch.randn(B, P, device=DEV, generator=g)
    t = (torch.rand(B * P, device=DEV, generator=g) < 0.07).to(torch.uint8)
    return x.to(torch.bfloat16).reshape(-1, 8), t


def _prep_net(case, seed):
    x, t = _net_inputs(case, seed)
    net = surrogate.UNet(case["B"], case["H"], case["W"], chans=_chans(case), seed=seed,
                         pos_weight=12.0, dice=1.0)
    return {"case": case, "net": net, "x": x, "t": t}


# -------------------------------------------------------------------- run
def run(st):
    return {"run": _run_run, "elastic": _run_elastic, "batch": _run_batch, "tri": _run_elastic,
            "layer": _run_layer, "infer": _run_infer, "grads": _run_grads}[st["case"]["kind"]](st)


def _run_run(st):
    s = st["solver"]
    s.load_state(st["blob"])
    s.step(st["case"]["steps"])
    n = s.prob.n_nodes
    f = s.nodes()
    return {"ux": f["ux"][:n], "uy": f["uy"][:n], "vx": f["vx"][:n], "vy": f["vy"][:n],
            "state": s.state()}


def _run_elastic(st):
    s = st["solver"]
    s.step(st["case"]["steps"])
    u, v = _fields(s, st["n"])
    return {"u": u, "v": v}


def _run_batch(st):
    members = st["members"]
    for m, blob in zip(members, st["blobs"]):
        m.load_state(blob)
    b = cem.Batch(members)
    b.step(st["case"]["steps"])
    b.close()
    u, state = [], []
    for m, n in zip(members, st["n"]):
        f = m.nodes()
        u += [f["ux"][:n], f["uy"][:n]]
        state.append(m.state())
    return {"u": np.concatenate(u), "state": np.concatenate(state)}


def _sg(rc, what):
    if rc != 0:
        raise RuntimeError(f"{what} failed with {rc}")


def _run_layer(st):
    L, c = surrogate.sg(), st["case"]
    B, H, W, cin, cout, pad = (c[k] for k in ("B", "H", "W", "cin", "cout", "pad"))
    s = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    p = lambda t: t.data_ptr()
    _sg(L.cem_sg_conv3x3(p(st["x"]), B, H, W, cin, cin, p(st["w"]), p(st["b"]), cout, 1, None, 0,
                         p(st["y"]), pad + cout, pad, s), "conv")
    _sg(L.cem_sg_conv3x3(p(st["dy"]), B, H, W, cout, cout, p(st["wt"]), None, cin, 0, p(st["x"]),
                         cin, p(st["dx"]), cin, 0, s), "data gradient")
    _sg(L.cem_sg_conv3x3_wgrad(p(st["x"]), cin, p(st["dy"]), cout, B, H, W, cin, cout,
                               p(st["dw"]), p(st["db"]), p(st["ws"]), st["ws_bytes"], s),
        "weight gradient")
    return {"y": st["y"][:, pad:], "dx": st["dx"], "dw": st["dw"], "db": st["db"]}


def _run_infer(st):
    net = st["net"]
    net.set_input(st["x"])
    return {"z": net.forward()}


def _run_grads(st):
    net = st["net"]
    net.set_input(st["x"])
    z = net.forward()
    loss = net.loss_and_grad(st["t"])
    net.backward()
    g = {n: [p["gw"], p["gb"]] for n, p in net.convs.items()}
    g["head"] = [net.head["gw"], net.head["gb"]]
    return {"z": z, "loss": loss, "grads": g}


# ------------------------------------------------------------------- work
def _sizes_batch(case):
    # mean of round(100 s) round(40 s), s uniform
    a, b = case["smin"], case["smax"]
    return int(case["count"] * 4000 * (b ** 3 - a ** 3) / (3 * (b - a)))


def work(case):
    """Bytes: per element-update 53 (FP32-mixed) or 73 (FP64): displacement
    and velocity read and written, the inverse mass and the element's state
    read; triangles also read their nodes and shape coefficients.  The
    convolutions: every tensor once.  Operations: the multiplications and
    additions of an element-update, two per multiply-add of a convolution."""
    k = case["kind"]
    if k in ("run", "elastic", "batch", "tri"):
        per = 53 if case["precision"] == FP32 else 73
        ne = {"run": lambda: case["nx"] * case["ny"], "elastic": lambda: case["n"] ** 2,
              "batch": lambda: _sizes_batch(case),
              "tri": lambda: 2 * case["nx"] * case["ny"]}[k]()
        if k == "tri":
            # half a node per triangle: 26.5 / 36.5 bytes, 3 node ids, 5 coefficients
            per = per // 2 + 12 + (20 if case["precision"] == FP32 else 40)
        return {"bytes": ne * case["steps"] * per + 32 * ne, "flops": ne * case["steps"] * 130}
    if k == "layer":
        P = case["B"] * case["H"] * case["W"]
        ci, co = case["cin"], case["cout"]
        # forward x, y; data gradient dy, mask, dx; weight gradient x, dy
        return {"bytes": 2 * P * (4 * ci + 3 * co) + 9 * ci * co * 8,
                "flops": 3 * 2 * 9 * P * ci * co}
    ch, flops, nbytes = _chans(case), 0, 0
    P = [case["B"] * (case["H"] >> l) * (case["W"] >> l) for l in range(case["levels"])]
    convs, c = [], 8
    for l, n in enumerate(ch):
        convs += [(P[l], c, n), (P[l], n, n)]
        c = n
    for l in range(case["levels"] - 2, -1, -1):
        convs += [(P[l], ch[l + 1] + ch[l], ch[l]), (P[l], ch[l], ch[l])]
    for p, ci, co in convs:
        flops += 2 * 9 * p * ci * co
        nbytes += 2 * p * (ci + co) + 18 * ci * co
    if k == "grads":
        flops, nbytes = 3 * flops - 2 * 9 * P[0] * 8 * ch[0], 3 * nbytes
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    k = case["kind"]
    if k == "elastic":
        return _exact_elastic(case, seed)
    if k == "tri":
        return _exact_tri(case, seed)
    if k == "layer":
        return _exact_layer(case, seed)
    if k in ("infer", "grads"):
        return _exact_net(case, seed, k == "grads")
    return None


def _law(bc, t):
    if bc.law == inputs.LAW_CONST:
        return 1.0
    if t <= bc.t0:
        return t / bc.t0
    return 1.0 if bc.law == inputs.LAW_RAMP else math.exp(-(t - bc.t0) / bc.tau)


def _elasticity(m):
    c = m.E / ((1 + m.nu) * (1 - 2 * m.nu))
    return c * (1 - m.nu), c * m.nu, c * (1 - 2 * m.nu) / 2


def _wave_speed(m):
    return math.sqrt(m.E * (1 - m.nu) / (m.rho * (1 + m.nu) * (1 - 2 * m.nu)))


def _exact_elastic(case, seed):
    """Bilinear quadrilaterals with strains at the edge midpoints, averaged
    across an edge between two active elements; central differences."""
    p = _elastic_problem(case, seed)
    n, h, m = case["n"], p.hx, p.material
    f8 = dict(dtype=torch.float64, device=DEV)
    act = torch.tensor(p.active.reshape(n, n), device=DEV).double()
    D11, D12, D33 = _elasticity(m)
    dt = 0.5 * h / _wave_speed(m)
    # derivatives of the shape functions of nodes 0..3 at edge points 0..3, in 1/(2h)
    NX = [[-2, 2, 0, 0], [-1, 1, 1, -1], [0, 0, 2, -2], [-1, 1, 1, -1]]
    NY = [[-1, -1, 1, 1], [0, -2, 2, 0], [-1, -1, 1, 1], [-2, 0, 0, 2]]
    q = 1.0 / (2 * h)
    F = np.zeros((2, (n + 1) * (n + 1)))
    bc = p.bcs[0]
    a = p.active.reshape(n, n)
    for e in bc.items.tolist():
        if e < n * (n + 1):
            j, i = divmod(e, n)
            up = j > 0 and a[j - 1, i]
            n1, n2, o = j * (n + 1) + i, j * (n + 1) + i + 1, (0.0, 1.0 if up else -1.0)
        else:
            j, i = divmod(e - n * (n + 1), n + 1)
            right = i > 0 and a[j, i - 1]
            n1, n2, o = j * (n + 1) + i, (j + 1) * (n + 1) + i, (1.0 if right else -1.0, 0.0)
        for N in (n1, n2):
            for c in (0, 1):
                F[c, N] -= 0.5 * h * bc.a0 * o[c]
    F = torch.tensor(F, **f8).view(2, n + 1, n + 1)
    mass = torch.zeros(n + 1, n + 1, **f8)
    corner = [(slice(0, n), slice(0, n)), (slice(0, n), slice(1, n + 1)),
              (slice(1, n + 1), slice(1, n + 1)), (slice(1, n + 1), slice(0, n))]
    for c in corner:
        mass[c] += m.rho * h * h / 4 * act
    minv = torch.where(mass > 0, 1 / mass, torch.zeros_like(mass))
    vx, vy = _modes(n, n, h, h, seed)
    v = torch.tensor(np.stack([vx, vy]), **f8).view(2, n + 1, n + 1)
    u = torch.zeros(2, n + 1, n + 1, **f8)
    bh = act[:-1, :] * act[1:, :]   # both sides of an inner horizontal edge
    bv = act[:, :-1] * act[:, 1:]
    for step in range(case["steps"]):
        un = [u[(slice(None),) + c] for c in corner]
        E = []
        for k in range(4):
            gx = sum(q * NX[k][s] * un[s] for s in range(4) if NX[k][s])
            gy = sum(q * NY[k][s] * un[s] for s in range(4) if NY[k][s])
            E.append(torch.stack([gx[0], gy[1], gy[0] + gx[1]]))
        d = 0.5 * bh * (E[0][:, 1:] - E[2][:, :-1])
        E[0][:, 1:] -= d
        E[2][:, :-1] += d
        d = 0.5 * bv * (E[3][:, :, 1:] - E[1][:, :, :-1])
        E[3][:, :, 1:] -= d
        E[1][:, :, :-1] += d
        fint = torch.zeros(2, n + 1, n + 1, **f8)
        for k in range(4):
            sx = (D11 * E[k][0] + D12 * E[k][1]) * act
            sy = (D12 * E[k][0] + D11 * E[k][1]) * act
            sxy = D33 * E[k][2] * act
            for s, c in enumerate(corner):
                w = h * h / 4 * q
                fint[(0,) + c] += w * (NX[k][s] * sx + NY[k][s] * sxy)
                fint[(1,) + c] += w * (NY[k][s] * sy + NX[k][s] * sxy)
        v = v + (0.5 * dt if step == 0 else dt) * (_law(bc, step * dt) * F - fint) * minv
        u = u + dt * v
    return {"u": u.reshape(-1), "v": v.reshape(-1)}


def _exact_tri(case, seed):
    """Constant-strain triangles: edge strains averaged by area, forces
    B^T sigma A/3 from every edge of every triangle; central differences."""
    p = _tri_problem(case, seed)
    m = p.material
    f8 = dict(dtype=torch.float64, device=DEV)
    X = torch.tensor(p.X, **f8)
    conn = torch.tensor(p.conn.astype(np.int64), device=DEV)
    ne, nn = len(p.conn), p.n_nodes
    ed = inputs.tri_edges(p.conn)
    e1 = torch.tensor(ed["e1"].astype(np.int64), device=DEV)
    e2 = torch.tensor(ed["e2"].astype(np.int64), device=DEV)
    two = e2 >= 0
    x, y = X[conn][..., 0], X[conn][..., 1]
    A2 = (x[:, 1] - x[:, 0]) * (y[:, 2] - y[:, 0]) - (x[:, 2] - x[:, 0]) * (y[:, 1] - y[:, 0])
    b = torch.stack([y[:, 1] - y[:, 2], y[:, 2] - y[:, 0], y[:, 0] - y[:, 1]], 1) / A2[:, None]
    c = torch.stack([x[:, 2] - x[:, 1], x[:, 0] - x[:, 2], x[:, 1] - x[:, 0]], 1) / A2[:, None]
    A = A2 / 2
    side = torch.stack([(X[conn[:, i]] - X[conn[:, (i + 1) % 3]]).norm(dim=1) for i in range(3)])
    hmin = float((A2 / side.max(0).values).min())
    dt = 0.5 * hmin / _wave_speed(m)
    D11, D12, D33 = _elasticity(m)
    mass = torch.zeros(nn, **f8)
    for i in range(3):
        mass.index_add_(0, conn[:, i], m.rho * A / 3)
    F = torch.zeros(2, nn, **f8)
    n1, n2 = (torch.tensor(ed[k].astype(np.int64), device=DEV) for k in ("n1", "n2"))
    for bc in p.bcs:
        it = torch.tensor(bc.items.astype(np.int64), device=DEV)
        half = 0.5 * (X[n1[it]] - X[n2[it]]).norm(dim=1) * bc.a0
        for N in (n1[it], n2[it]):
            F[1].index_add_(0, N, half)
    w1, w2 = A[e1], torch.where(two, A[e2.clamp(min=0)], torch.zeros_like(A[e1]))
    u = torch.tensor(np.stack(p.init[:2]), **f8)
    v = torch.tensor(np.stack(p.init[2:]), **f8)
    for step in range(case["steps"]):
        un = u[:, conn]
        exx, eyy = (b * un[0]).sum(1), (c * un[1]).sum(1)
        gxy = (c * un[0]).sum(1) + (b * un[1]).sum(1)
        eps = torch.stack([exx, eyy, gxy])
        sm = (w1 * eps[:, e1] + w2 * eps[:, e2.clamp(min=0)]) / (w1 + w2)
        # the stresses of a triangle's three edges, summed
        tot = torch.zeros(3, ne, **f8)
        tot.index_add_(1, e1, sm)
        tot.index_add_(1, e2[two], sm[:, two])
        sx, sy = D11 * tot[0] + D12 * tot[1], D12 * tot[0] + D11 * tot[1]
        sxy = D33 * tot[2]
        fint = torch.zeros(2, nn, **f8)
        for i in range(3):
            fint[0].index_add_(0, conn[:, i], (b[:, i] * sx + c[:, i] * sxy) * A / 3)
            fint[1].index_add_(0, conn[:, i], (c[:, i] * sy + b[:, i] * sxy) * A / 3)
        v = v + (0.5 * dt if step == 0 else dt) * (F - fint) / mass
        u = u + dt * v
    return {"u": u.reshape(-1), "v": v.reshape(-1)}


def _taps(B, H, W):
    """For each tap (ky, kx): the output and input windows it joins."""
    for ky in range(3):
        for kx in range(3):
            o = (slice(None), slice(max(0, 1 - ky), min(H, H + 1 - ky)),
                 slice(max(0, 1 - kx), min(W, W + 1 - kx)))
            i = (slice(None), slice(max(0, ky - 1), min(H, H + ky - 1)),
                 slice(max(0, kx - 1), min(W, W + kx - 1)))
            yield ky, kx, o, i


def _conv64(x, w, b):
    B, H, W, _ = x.shape
    y = b.expand(B, H, W, -1).clone()
    for ky, kx, o, i in _taps(B, H, W):
        y[o] += x[i] @ w[:, ky, kx].T
    return y


def _conv64_bwd(x, w, dy):
    B, H, W, ci = x.shape
    dw, dx = torch.zeros_like(w), torch.zeros_like(x)
    for ky, kx, o, i in _taps(B, H, W):
        dw[:, ky, kx] = dy[o].reshape(-1, dy.shape[3]).T @ x[i].reshape(-1, ci)
        dx[i] += dy[o] @ w[:, ky, kx]
    return dx, dw, dy.sum((0, 1, 2))


def _exact_layer(case, seed):
    x, dy, w, b = _layer_tensors(case, seed)
    B, H, W, cin, cout = (case[k] for k in ("B", "H", "W", "cin", "cout"))
    P = B * H * W
    x, dy = x.double().view(B, H, W, cin), dy.double().view(B, H, W, cout)
    w, b = w.double(), b.double()
    y = _conv64(x, w, b).clamp_(min=0)
    dx, dw, db = _conv64_bwd(x, w, dy)
    return {"y": y.reshape(P, cout), "dx": (dx * (x > 0)).reshape(P, cin), "dw": dw, "db": db}


def _net_weights(case, seed):
    """The network's initial weights: scaled normal draws in layer order."""
    rng, ch, w, c = np.random.default_rng(seed), _chans(case), {}, 8
    order = []
    for l, n in enumerate(ch):
        order += [(f"e{l}a", c, n), (f"e{l}b", n, n)]
        c = n
    for l in range(len(ch) - 2, -1, -1):
        order += [(f"d{l}a", ch[l + 1] + ch[l], ch[l]), (f"d{l}b", ch[l], ch[l])]
    for name, ci, co in order:
        v = rng.standard_normal((co, 3, 3, ci)) * math.sqrt(2.0 / (9 * (3 if name == "e0a" else ci)))
        if name == "e0a":
            v[..., 3:] = 0.0
        w[name] = torch.tensor(v, dtype=torch.float32, device=DEV).double()
    head = rng.standard_normal(ch[0]) * math.sqrt(2.0 / ch[0]) * 0.1
    return w, torch.tensor(head, dtype=torch.float32, device=DEV).double()


def _exact_net(case, seed, grads):
    B, H, W, L = case["B"], case["H"], case["W"], case["levels"]
    xin, t = _net_inputs(case, seed)
    w, hw = _net_weights(case, seed)
    zero = lambda n: torch.zeros(n, dtype=torch.float64, device=DEV)
    zs, bce, dice = [], 0.0, 0.0
    n_all, pw = B * H * W, 12.0
    for k in range(B):  # image by image: nothing couples them but the sums
        x = xin.view(B, H, W, 8)[k:k + 1].double()
        skip = []
        conv = lambda name, a: _conv64(a, w[name], zero(w[name].shape[0])).clamp_(min=0)
        h = x
        for l in range(L):
            s = conv(f"e{l}b", conv(f"e{l}a", h))
            skip.append(s)
            if l < L - 1:
                _, hh, ww, cc = s.shape
                h = s.view(1, hh // 2, 2, ww // 2, 2, cc).amax((2, 4))
        h = s
        for l in range(L - 2, -1, -1):
            up = h.repeat_interleave(2, 1).repeat_interleave(2, 2)
            cat = torch.cat([up, skip[l]], 3)
            h = conv(f"d{l}b", conv(f"d{l}a", cat))
        z = (h @ hw).reshape(-1)
        zs.append(z)
        if not grads:
            continue
        tt = t.view(B, -1)[k].double()
        sig = torch.sigmoid(z)
        sp = torch.nn.functional.softplus
        bce += float((pw * tt * sp(-z) + (1 - tt) * sp(z)).sum()) / n_all
        I, S = (sig * tt).sum(), sig.sum() + tt.sum()
        dice += float(1 - (2 * I + 1) / (S + 1)) / B
    out = {"z": torch.cat(zs)}
    if grads:
        out["loss"] = torch.tensor([bce, dice], dtype=torch.float64)
        # the gradients pass through every pooling's choice of its maximum, which
        # BF16 activations tie or swap: no 64-bit value to hold them to
        out["grads"] = None
    return out
