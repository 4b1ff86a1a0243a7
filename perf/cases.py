"""Work that users of this package have it do, with inputs, sizes and exact values.

Every case goes through the public bindings (lbm, fno, ffno, unet):
  lbm       one lattice: back to rest, started from a given flow (a surrogate's prediction), stepped,
            its time average and force rows read
  batch     several uneven channels stepped together from given flows, their averages on the surrogate's grid
  resample  a mean field onto the surrogate's grid
  fno       forward, or one training step, of the Fourier surrogate (BF16 activations)
  ffno      forward, or one training step, of the factorised surrogate (FP32)
  conv      one 3x3x3 convolution layer of the U-Net: forward, or its two gradients
"""
import math

import numpy as np
import torch

from paper_2606_16765_gb300 import ffno as FF
from paper_2606_16765_gb300 import fno as F
from paper_2606_16765_gb300 import inputs as I
from paper_2606_16765_gb300 import lbm as B
from paper_2606_16765_gb300 import unet as U

SURROGATE = (128, 64, 64)           # the surrogate's grid (x, y, z)
U_IN = 0.05
LBM_BYTES = {"f64": 8, "f32": 4, "f16s": 2, "f16c": 2}


def listed():
    return [
        # the small sphere channel of the parity runs: start-up of a lattice, every launch counts
        dict(name="lbm_sphere_small", kind="lbm", nx=64, ny=32, nz=32, body="sphere", storage="f32", steps=100,
             mean_every=10),
        # the cylinder channel whose lift and drag are recorded
        dict(name="lbm_cylinder", kind="lbm", nx=256, ny=128, nz=128, body="cylinder", storage="f32", steps=40,
             mean_every=10),
        # half the linear size of the full composite channel, 16-bit populations: a production run's step
        dict(name="lbm_composite", kind="lbm", nx=512, ny=256, nz=256, body="composite", storage="f16s", steps=20,
             mean_every=10),
        # the data pipeline: uneven channels of the training set stepped as one batch
        dict(name="batch_channels", kind="batch", members=8, storage="f16c", steps=20),
        # one member's mean field on its way into the training set
        dict(name="resample_mean", kind="resample", nx=192, ny=128, nz=96, mx=128, my=64, mz=64),
        # the surrogate's prediction for a batch of geometries
        dict(name="fno_predict", kind="fno", do="forward", batch=8, nx=128, ny=64, nz=64, mx=16, my=8, mz=8, layers=4,
             width=32),
        # one step of its training
        dict(name="fno_train", kind="fno", do="train", batch=8, nx=128, ny=64, nz=64, mx=16, my=8, mz=8, layers=4,
             width=32),
        # the factorised surrogate: one geometry, as in a design loop
        dict(name="ffno_predict", kind="ffno", do="forward", batch=1, nx=128, ny=64, nz=64, mx=32, my=16, mz=16,
             layers=4, width=32),
        # one step of its training
        dict(name="ffno_train", kind="ffno", do="train", batch=8, nx=128, ny=64, nz=64, mx=32, my=16, mz=16, layers=4,
             width=32),
        # U-Net layers: the first stage's second convolution on the full grid,
        dict(name="conv_top", kind="conv", do="forward", batch=4, nx=128, ny=64, nz=64, cin=32, cout=32),
        # the gradients of the second stage's second convolution,
        dict(name="conv_mid_grad", kind="conv", do="backward", batch=8, nx=64, ny=32, nz=32, cin=64, cout=64),
        # and a small call: the way into the bottleneck for a few samples
        dict(name="conv_deep", kind="conv", do="forward", batch=2, nx=8, ny=4, nz=4, cin=256, cout=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _draw(rng)
        if case not in known:
            return case


def _draw(rng):
    kind = rng.choice(["lbm", "lbm", "batch", "resample", "fno", "ffno", "ffno", "conv", "conv"])
    if kind == "lbm":
        nx, ny, nz = _log_int(rng, 48, 384), _log_int(rng, 24, 192), _log_int(rng, 24, 192)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, body=rng.choice(["sphere", "cylinder", "composite"]),
                    storage=rng.choice(["f64", "f32", "f32", "f16s", "f16c"]), steps=2 * rng.randint(5, 25),
                    mean_every=rng.choice([5, 10]))
    if kind == "batch":
        return dict(kind=kind, members=rng.randint(2, 10), storage=rng.choice(["f32", "f16s", "f16c"]),
                    steps=10 * rng.randint(1, 3))
    if kind == "resample":
        return dict(kind=kind, nx=_log_int(rng, 64, 512), ny=_log_int(rng, 32, 256), nz=_log_int(rng, 32, 256),
                    mx=rng.choice([64, 128, 200]), my=rng.choice([32, 64, 100]), mz=rng.choice([32, 64, 100]))
    if kind == "fno":
        nx, ny, nz = rng.choice([(128, 64, 64), (128, 64, 64), (128, 32, 64), (64, 64, 64), (96, 48, 48)])
        return dict(kind=kind, do=rng.choice(["forward", "train"]), batch=rng.randint(1, 8), nx=nx, ny=ny, nz=nz,
                    mx=16, my=8, mz=8, layers=rng.randint(1, 4), width=32)
    if kind == "ffno":
        nx, ny, nz = rng.choice([(128, 64, 64), (128, 64, 64), (64, 64, 64), (128, 32, 48), (96, 48, 64), (75, 50, 33)])
        return dict(kind=kind, do=rng.choice(["forward", "train"]), batch=rng.randint(1, 8), nx=nx, ny=ny, nz=nz,
                    mx=rng.choice([16, 24, 32]), my=rng.choice([8, 12, 16]), mz=rng.choice([8, 12, 16]),
                    layers=rng.randint(1, 4), width=rng.choice([32, 32, 20]))
    level = rng.randint(0, 4)
    ch = [32, 64, 128, 256, 512]
    cin = rng.choice([ch[level], ch[max(0, level - 1)], ch[level] + ch[min(4, level + 1)]])
    do = rng.choice(["forward", "backward"])
    return dict(kind="conv", do=do, batch=rng.randint(1, 4 if level == 0 else 8), nx=128 >> level, ny=64 >> level,
                nz=64 >> level, cin=cin, cout=ch[level])


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(1 + seed)


def _body(case, seed):
    grid = (case["nx"], case["ny"], case["nz"])
    nx, ny, nz = grid
    if case["body"] == "sphere":
        return I.sphere(grid, (0.25 * nx, 0.5 * (ny - 1), 0.5 * (nz - 1)), min(ny, nz) / 8.0), min(ny, nz) / 4.0
    if case["body"] == "cylinder":
        return I.cylinder_z(grid, (0.25 * nx, 0.5 * (ny - 1)), ny / 8.0), ny / 8.0
    s = ny / 512.0
    obs = I.composite(seed, grid, size_range=(max(6.0, 20.0 * s), max(6.0, 60.0 * s)), jitter=10.0 * s)
    return obs.mask(), float(ny)


def _flow(grid, mask, seed):
    """A flow as a surrogate predicts it: (u, v, w, p) [nz, ny, nx, 4], the channel stream with smooth deviations."""
    nx, ny, nz = grid
    g = _gen(seed)
    a = torch.rand((4, 6), generator=g, device="cuda", dtype=torch.float64)
    x = torch.arange(nx, device="cuda", dtype=torch.float64).view(1, 1, nx) / nx
    y = torch.arange(ny, device="cuda", dtype=torch.float64).view(1, ny, 1) / ny
    z = torch.arange(nz, device="cuda", dtype=torch.float64).view(nz, 1, 1) / nz
    f = torch.zeros((nz, ny, nx, 4), device="cuda", dtype=torch.float32)
    for c in range(4):
        k = [2.0 * math.pi * (1 + int(3 * float(v))) for v in a[c, :3]]
        ph = [2.0 * math.pi * float(v) for v in a[c, 3:]]
        w = torch.sin(k[0] * x + ph[0]) * torch.sin(k[1] * y + ph[1]) * torch.sin(k[2] * z + ph[2])
        f[..., c] = (0.15 * U_IN * w if c < 3 else 2e-4 * w).float()
    f[..., 0] += U_IN
    f[torch.from_numpy(mask).cuda() != 0] = 0.0
    return f


def _lbm_params(case, l_ref, re):
    return dict(storage=case["storage"], re=re, u_in=U_IN, l_ref=l_ref, mean_start=0, mean_end=1 << 40,
                mean_every=case.get("mean_every", 10))


def _batch_members(case, seed):
    """Channels as the training set draws them: uneven grids, Re log-uniform, a composite obstacle each.  The sizes
    go round so that a batch of n costs the same for every seed."""
    rng = np.random.default_rng(77 + seed)
    out = []
    for g in range(case["members"]):
        grid = ((128, 192, 256)[g % 3], (64, 96, 128)[(g // 3) % 3], (96, 64, 128)[g % 3])
        s = grid[1] / 512.0
        obs = I.composite(1000 * seed + g, grid, size_range=(max(6.0, 20.0 * s), max(6.0, 60.0 * s)), jitter=10.0 * s)
        out.append((grid, obs.mask(), float(math.exp(rng.uniform(math.log(1e3), math.log(1e4))))))
    return out


def _net_shapes(case):
    """(name, shape, bound of the uniform distribution) of the parameters in the flat vector's order."""
    W, L, cin, cout, hidden, lift = case["width"], case["layers"], 4, 4, 128, 32
    s = []

    def linear(name, o, i):
        s.extend([(name + "w", (o, i), 1 / math.sqrt(i)), (name + "b", (o,), 1 / math.sqrt(i))])

    if case["kind"] == "fno":
        for l in range(L):
            s.append((f"R{l}", (case["mz"], 2 * case["my"], 2 * case["mx"], W, W, 2), 1.0 / (W * W)))
    linear("P1", lift, cin)
    linear("P2", W, lift)
    for l in range(L):
        if case["kind"] == "fno":
            linear(f"W{l}", W, W)
        else:
            s.extend((f"R{l}{d}", (W, W, case["m" + d], 2), 1.0 / (W * W)) for d in "zyx")
            linear(f"Fa{l}", W, W)
            linear(f"Fb{l}", W, W)
    s.extend([("Q1w", (hidden, W), 1.0 / W), ("Q1b", (hidden,), 1 / math.sqrt(W)),
              ("Q2w", (cout, hidden), math.sqrt(6.0 / hidden) / 30.0), ("Q2b", (cout,), 1 / math.sqrt(hidden))])
    return s


def _net_inputs(case, seed):
    """Parameters (flat, FP32), features, targets and loss weights on the device."""
    g = _gen(seed)
    u = lambda shape: torch.rand(shape, generator=g, device="cuda")  # noqa: E731
    p = torch.cat([((2 * u((math.prod(shape),)) - 1) * b) for _, shape, b in _net_shapes(case)])
    nb, nx, ny, nz = case["batch"], case["nx"], case["ny"], case["nz"]
    # mask of a body, log10 Re - 3.5, cos and sin of the angle of attack
    x = torch.zeros((nb, 4, nz, ny, nx), device="cuda")
    sol = u((nb, 3)).tolist()
    for b in range(nb):
        x0, y0, z0 = (int(n * (0.25 + 0.2 * v)) for n, v in zip((nx, ny, nz), sol[b]))
        x[b, 0, z0:z0 + nz // 5, y0:y0 + ny // 4, x0:x0 + nx // 8] = 1.0
    re, al = u((nb, 1, 1, 1)) - 0.5, (u((nb, 1, 1, 1)) - 0.5) * math.pi / 3
    x[:, 1], x[:, 2], x[:, 3] = re, torch.cos(al), torch.sin(al)
    t = 0.5 + 0.3 * torch.randn((nb, 4, nz // 8 + 1, ny // 8 + 1, nx // 8 + 1), generator=g, device="cuda")
    t = torch.nn.functional.interpolate(t, size=(nz, ny, nx), mode="trilinear").contiguous()
    m = torch.zeros((nb, nz, ny, nx), device="cuda")
    m[:, nz // 4:3 * nz // 4, ny // 4:3 * ny // 4, nx // 10:9 * nx // 10] = 1.0
    m *= x[:, 0] == 0
    return p, x, t, m


def _conv_inputs(case, seed):
    """Activations after a ReLU, an output gradient and He-scaled weights, on the values BF16 has: what the U-Net
    stores between its layers."""
    g = _gen(seed)
    nb, nx, ny, nz, ci, co = (case[k] for k in ("batch", "nx", "ny", "nz", "cin", "cout"))
    r = lambda *s: torch.randn(s, generator=g, device="cuda")  # noqa: E731
    w = (r(co, ci, 27) * math.sqrt(2.0 / (27 * ci))).bfloat16().float()
    x = r(nb, nz, ny, nx, ci).clamp_min_(0).bfloat16().float()
    gy = r(nb, nz, ny, nx, co).bfloat16().float() if case["do"] == "backward" else None
    return x, w, gy


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lbm":
        mask, l_ref = _body(case, seed)
        grid = (case["nx"], case["ny"], case["nz"])
        s = B.Solver(grid, mask, force_every=1, **_lbm_params(case, l_ref, 1000.0 + 10.0 * (seed % 300)))
        mean = torch.empty(s.shape + (4,), device="cuda", dtype=torch.float64 if case["storage"] == "f64"
                           else torch.float32)
        return dict(case=case, solver=s, flow=_flow(grid, mask, seed), mean=mean)
    if kind == "batch":
        mem = _batch_members(case, seed)
        b = B.Batch([dict(grid=grid, mask=mask, **_lbm_params(case, float(grid[1]), re)) for grid, mask, re in mem])
        b.set_end([1 << 40] * len(mem))
        mx, my, mz = SURROGATE
        bufs = []
        for k, (grid, mask, _) in enumerate(mem):
            b.member(k).init_equilibrium(_flow(grid, mask, seed + k))
            bufs.append(torch.empty((grid[2], grid[1], grid[0], 4), device="cuda"))
        return dict(case=case, batch=b, members=[b.member(k) for k in range(len(mem))], bufs=bufs,
                    out=torch.empty((len(mem), 4, mz, my, mx), device="cuda"))
    if kind == "resample":
        grid = (case["nx"], case["ny"], case["nz"])
        mask = I.composite(seed, grid, size_range=(6.0, 12.0), jitter=2.0).mask()
        return dict(case=case, src=_flow(grid, mask, seed),
                    out=torch.empty((4, case["mz"], case["my"], case["mx"]), device="cuda"))
    if kind in ("fno", "ffno"):
        p, x, t, m = _net_inputs(case, seed)
        cfg = {k: case[k] for k in ("nx", "ny", "nz", "mx", "my", "mz", "layers", "width")}
        if kind == "fno":
            net = F.FNO(max_batch=case["batch"], **cfg)
        else:
            net = FF.FFNO(max_batch=case["batch"], ff_hidden=case["width"], **cfg)
        net.set_params(p.cpu().numpy())
        if case["do"] == "forward":
            return dict(case=case, net=net, x=x, y=torch.empty_like(t))
        return dict(case=case, net=net, x=x, t=t, m=m, grads=torch.empty_like(p))
    x, w, gy = _conv_inputs(case, seed)
    if case["do"] == "forward":
        return dict(case=case, x=x, w=w, y=torch.empty(x.shape[:4] + (case["cout"],), device="cuda"))
    return dict(case=case, x=x, w=w, gy=gy, gx=torch.empty_like(x), gw=torch.empty_like(w))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case = state["case"]
    kind = case["kind"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "lbm":
        s = state["solver"]
        s.reset()
        s.init_equilibrium(state["flow"])
        s.step(case["steps"])
        B.lbm_read_mean(s.h, state["mean"], 0 if case["storage"] == "f64" else 1, 0)
        # momentum exchange of populations kept to FP32 at most carries no more digits than that
        return {"mean": state["mean"], "forces": s.forces().astype(np.float32)}
    if kind == "batch":
        state["batch"].run(case["steps"])
        for k, m in enumerate(state["members"]):
            B.lbm_read_mean(m.h, state["bufs"][k], 1, 0)
            B.lbm_resample(state["bufs"][k], (m.grid.nx, m.grid.ny, m.grid.nz), 4, 0, state["out"][k], SURROGATE,
                           stream)
        return state["out"]
    if kind == "resample":
        B.lbm_resample(state["src"], (case["nx"], case["ny"], case["nz"]), 4, 0, state["out"],
                       (case["mx"], case["my"], case["mz"]), stream)
        return state["out"]
    if kind == "conv":
        if case["do"] == "forward":
            U.conv3_forward(state["x"], state["w"], state["y"], stream)
            return state["y"]
        U.conv3_backward_data(state["gy"], state["w"], state["gx"], stream)
        U.conv3_backward_weights(state["x"], state["gy"], state["gw"], stream)
        return {"gx": state["gx"], "gw": state["gw"]}
    net = state["net"]
    if case["do"] == "forward":
        return net.forward(state["x"], state["y"])
    # the end of the cosine schedule: the rate tends to 0 and the parameters stay where they are
    if kind == "fno":
        loss = net.train_step(state["x"], state["t"], state["m"], 1e-7)
        F.fno_get_grads(net.h, state["grads"])
        return {"loss": loss, "grads": state["grads"]}
    loss = net.loss_grad(state["x"], state["t"], state["m"])
    net.adam(1e-7)
    return {"loss": loss, "grads": net.grads()}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind in ("lbm", "batch"):
        if kind == "lbm":
            cells = case["nx"] * case["ny"] * case["nz"]
            io = cells * (16 + (32 if case["storage"] == "f64" else 16))
        else:
            cells = sum(math.prod(((128, 192, 256)[g % 3], (64, 96, 128)[(g // 3) % 3], (96, 64, 128)[g % 3]))
                        for g in range(case["members"]))
            io = case["members"] * 16 * math.prod(SURROGATE)
        samples = -(-case["steps"] // case.get("mean_every", 10))
        # populations once in and once out per step; FP64 running sums per averaged sample
        return {"bytes": cells * (54 * LBM_BYTES[case["storage"]] * case["steps"] + 64 * samples) + io,
                "flops": cells * 900 * case["steps"]}
    if kind == "resample":
        n, m = case["nx"] * case["ny"] * case["nz"], case["mx"] * case["my"] * case["mz"]
        return {"bytes": 16 * (n + m), "flops": 4 * 24 * m}
    cells = case["batch"] * case["nx"] * case["ny"] * case["nz"]
    if kind == "conv":
        ci, co = case["cin"], case["cout"]
        mac = 27 * ci * co
        if case["do"] == "forward":
            return {"bytes": 4 * (cells * (ci + co) + mac), "flops": 2 * mac * cells}
        return {"bytes": 4 * (cells * (2 * ci + co) + 2 * mac), "flops": 4 * mac * cells}
    W, L = case["width"], case["layers"]
    # one pointwise pass of the network; fast transforms (5/2 n log2 n per line); the contraction of the kept modes
    point = 2 * (4 * 32 + 32 * W + L * W * W * (1 if kind == "fno" else 2) + W * 128 + 128 * 4)
    lines = sum(math.log2(case[n]) for n in ("nx", "ny", "nz"))
    if kind == "fno":
        modes = case["batch"] * case["mz"] * 4 * case["my"] * case["mx"]
    else:
        modes = cells * sum(case[m] / case[n] for m, n in (("mx", "nx"), ("my", "ny"), ("mz", "nz")))
    flops = cells * (point + L * W * 2 * 2.5 * lines) + L * modes * 8 * W * W
    params = sum(math.prod(s) for _, s, _ in _net_shapes(case))
    if case["do"] == "forward":
        return {"bytes": 4 * (8 * cells + params), "flops": flops}
    return {"bytes": 4 * (9 * cells + 8 * params), "flops": 3 * flops}


# ---------------------------------------------------------------------------
# exact values, in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind == "lbm":
        mask, l_ref = _body(case, seed)
        grid = (case["nx"], case["ny"], case["nz"])
        mean, forces = _lattice(case, grid, mask, l_ref, 1000.0 + 10.0 * (seed % 300), _flow(grid, mask, seed))
        return {"mean": mean, "forces": forces}
    if kind == "batch":
        out = []
        for k, (grid, mask, re) in enumerate(_batch_members(case, seed)):
            mean, _ = _lattice(case, grid, mask, float(grid[1]), re, _flow(grid, mask, seed + k))
            out.append(_resample(mean, SURROGATE))
        return torch.stack(out)
    if kind == "resample":
        grid = (case["nx"], case["ny"], case["nz"])
        mask = I.composite(seed, grid, size_range=(6.0, 12.0), jitter=2.0).mask()
        return _resample(_flow(grid, mask, seed).double(), (case["mx"], case["my"], case["mz"]))
    if kind == "conv":
        x, w, gy = _conv_inputs(case, seed)
        w = w.double()
        if case["do"] == "forward":
            return _conv(x, w.permute(2, 1, 0))
        return {"gx": _conv(gy, w.flip(2).permute(2, 0, 1)), "gw": _conv_gw(x, gy)}
    return _net(case, seed)


def _shifted(x, tap):
    """x [B, z, y, x, c] with a zero border, moved so that cell n holds its neighbour n + tap - 1."""
    nz, ny, nx = x.shape[1:4]
    p = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    a, b, c = tap // 9, (tap // 3) % 3, tap % 3
    return p[:, a:a + nz, b:b + ny, c:c + nx]


def _conv(x, w):
    """Sum over the taps of shifted x times w [27, in, out]; one sample after the other."""
    out = []
    for b in range(x.shape[0]):
        xb = x[b:b + 1].double()
        y = torch.zeros(xb.shape[:4] + (w.shape[2],), device="cuda", dtype=torch.float64)
        for tap in range(27):
            y += _shifted(xb, tap) @ w[tap]
        out.append(y)
    return torch.cat(out)


def _conv_gw(x, gy):
    ci, co = x.shape[-1], gy.shape[-1]
    gw = torch.zeros((co, ci, 27), device="cuda", dtype=torch.float64)
    for b in range(x.shape[0]):
        xb, gb = x[b:b + 1].double(), gy[b].reshape(-1, co).double()
        for tap in range(27):
            gw[:, :, tap] += gb.T @ _shifted(xb, tap).reshape(-1, ci)
    return gw


def _resample(src, grid):
    """src [z, y, x, c] -> [c, mz, my, mx]: cell-centred, linear along each axis."""
    t = src.permute(3, 0, 1, 2)
    for ax, m in zip((3, 2, 1), grid):
        n = t.shape[ax]
        s = ((torch.arange(m, device="cuda", dtype=torch.float64) + 0.5) * n / m - 0.5).clamp(0, n - 1)
        i0 = s.floor().long()
        shape = [1, 1, 1, 1]
        shape[ax] = m
        w = (s - i0).view(shape)
        t = t.index_select(ax, i0) * (1 - w) + t.index_select(ax, (i0 + 1).clamp(max=n - 1)) * w
    return t.contiguous()


def _net(case, seed):
    """Both networks in complex128, one sample at a time; gradients by autograd."""
    p, x, t, m = _net_inputs(case, seed)
    P, o = {}, 0
    for name, shape, _ in _net_shapes(case):
        n = math.prod(shape)
        P[name] = p[o:o + n].view(shape).double().requires_grad_(case["do"] == "train")
        o += n
    nx, ny, nz, mx, my, mz = (case[k] for k in ("nx", "ny", "nz", "mx", "my", "mz"))
    gelu = torch.nn.functional.gelu
    lin = lambda n, v: torch.einsum("oi,bizyx->bozyx", P[n + "w"], v) + P[n + "b"].view(1, -1, 1, 1, 1)  # noqa: E731

    def fourier(v, l):
        f = torch.fft.fftn(torch.fft.rfft(v, dim=2)[:, :, :mz], dim=(3, 4))
        jy, jx = list(range(my)) + list(range(ny - my, ny)), list(range(mx)) + list(range(nx - mx, nx))
        f = f[:, :, :, jy][..., jx]
        g = torch.einsum("bizyx,zyxio->bozyx", f, torch.view_as_complex(P[f"R{l}"]))
        full = torch.zeros(v.shape[:2] + (nz // 2 + 1, ny, nx), device="cuda", dtype=g.dtype)
        at = [torch.tensor(k, device="cuda").view(s) for k, s in ((range(mz), (-1, 1, 1)), (jy, (1, -1, 1)),
                                                                   (jx, (1, 1, -1)))]
        full = full.index_put((torch.arange(full.shape[0], device="cuda").view(-1, 1, 1, 1, 1),
                               torch.arange(full.shape[1], device="cuda").view(1, -1, 1, 1, 1), *at), g)
        return torch.fft.irfft(torch.fft.ifftn(full, dim=(3, 4)), n=nz, dim=2)

    def factorised(v, l):
        u = 0
        for d, ax, n, k in (("z", 2, nz, mz), ("y", 3, ny, my), ("x", 4, nx, mx)):
            f = torch.fft.rfft(v, dim=ax).narrow(ax, 0, k).movedim(ax, -1)
            g = torch.einsum("biyxk,iok->boyxk", f, torch.view_as_complex(P[f"R{l}{d}"]))
            u = u + torch.fft.irfft(g, n=n, dim=-1).movedim(-1, ax)
        return u

    def net(x):
        v = lin("P2", gelu(lin("P1", x)))
        for l in range(case["layers"]):
            if case["kind"] == "fno":
                v = fourier(v, l) + lin(f"W{l}", v)
                v = gelu(v) if l < case["layers"] - 1 else v
            else:
                v = v + lin(f"Fb{l}", gelu(lin(f"Fa{l}", factorised(v, l))))
        return lin("Q2", torch.sin(30.0 * lin("Q1", v)))

    ys, loss = [], 0.0
    for b in range(case["batch"]):
        y = net(x[b:b + 1].double())
        if case["do"] == "forward":
            ys.append(y)
            continue
        e = (m[b:b + 1, None].double() * (y - t[b:b + 1].double()) ** 2).sum() / (4 * m.double().sum())
        e.backward()
        loss += float(e.detach())
    if case["do"] == "forward":
        return torch.cat(ys)
    return {"loss": torch.tensor(loss, dtype=torch.float64),
            "grads": torch.cat([P[n].grad.reshape(-1) for n, _, _ in _net_shapes(case)])}


C = [(i % 3 - 1, (i // 3) % 3 - 1, i // 9 - 1) for i in range(27)]      # velocities
WT = [(8 / 27, 2 / 27, 1 / 54, 1 / 216)[sum(map(abs, c))] for c in C]   # weights


def _lattice(case, grid, mask, l_ref, re, flow):
    """The channel in FP64: cumulant collision (rates of the shear and of all else, Galilean-corrected), two arrays
    and pull streaming, moving-wall inlet, convective outflow, halfway bounce-back.  (mean [z, y, x, 4], forces)."""
    if math.prod(grid) * case["steps"] > 9e8:
        return None, None                                              # beyond about twenty seconds
    nx, ny, nz = grid
    w1 = 1.0 / (3.0 * U_IN * l_ref / re + 0.5)
    solid = torch.from_numpy(mask).cuda() != 0
    one = lambda c, v: 2.0 / 3.0 - v * v if c == 0 else 0.5 * (1.0 / 3.0 + v * v + c * v)  # noqa: E731
    fl = flow.double()
    f = torch.empty((27, nz, ny, nx), device="cuda", dtype=torch.float64)
    for i, (cx, cy, cz) in enumerate(C):
        f[i] = (1.0 + 3.0 * fl[..., 3]) * one(cx, fl[..., 0]) * one(cy, fl[..., 1]) * one(cz, fl[..., 2])
        f[i][solid] = WT[i]
    fluid = (~solid).double()
    mean, samples, forces = torch.zeros((nz, ny, nx, 4), device="cuda", dtype=torch.float64), 0, []
    # obstacle links: fluid cells whose neighbour along c_i is solid and inside the grid
    pad = torch.nn.functional.pad(solid, (1, 1, 1, 1, 1, 1))
    link = [pad[1 + c[2]:1 + c[2] + nz, 1 + c[1]:1 + c[1] + ny, 1 + c[0]:1 + c[0] + nx] & ~solid for c in C]
    links = [torch.nonzero(k.reshape(-1)).view(-1) for k in link]
    for t in range(case["steps"]):
        post, rho, u = _collide(f, w1)
        if t % case.get("mean_every", 10) == 0:
            for d in range(3):
                mean[..., d] += u[d] * fluid
            mean[..., 3] += (rho - 1.0) / 3.0 * fluid
            samples += 1
        out = torch.stack([post[i].reshape(-1)[links[i]].sum() for i in range(27)])
        forces.append(torch.stack([2.0 * sum(C[i][d] * out[i] for i in range(27)) for d in range(3)]))
        new = torch.empty_like(f)
        for i, (cx, cy, cz) in enumerate(C):
            j = 26 - i
            v = post[j].clone()                                        # every link that ends at a wall comes back
            sx, sy, sz = ((max(0, c), n + min(0, c)) for c, n in zip((cx, cy, cz), grid))
            dst = (slice(*sz), slice(*sy), slice(*sx))
            src = (slice(sz[0] - cz, sz[1] - cz), slice(sy[0] - cy, sy[1] - cy), slice(sx[0] - cx, sx[1] - cx))
            v[dst] = torch.where(solid[src], v[dst], post[i][src])
            lat = (slice(*sz), slice(*sy))                             # not beyond a lateral wall
            if cx == 1:
                v[lat + (0,)] = post[j][lat + (0,)] + 6.0 * WT[i] * U_IN
            if cx == -1:
                cs = 1.0 / math.sqrt(3.0)
                inner = torch.where(solid[lat + (nx - 2,)], f[i][lat + (nx - 1,)], f[i][lat + (nx - 2,)])
                v[lat + (nx - 1,)] = cs * inner + (1.0 - cs) * f[i][lat + (nx - 1,)]
            v[solid] = WT[i]
            new[i] = v
        f = new
    return mean / samples, torch.stack(forces)


def _collide(f, w1):
    rho = f.sum(0)
    u = [sum(C[i][d] * f[i] for i in range(27)) / rho for d in range(3)]
    # central moments: the three axes one after the other, (c - u)^a summed over c
    k = {(c[0], c[1], c[2]): f[i] / rho for i, c in enumerate(C)}
    for d in range(3):
        low, mid, up = ((-1.0 - u[d]), -u[d], (1.0 - u[d]))
        new = {}
        for key in k:
            if key[d] != 0:
                continue
            a, b, c = (k[key[:d] + (s,) + key[d + 1:]] for s in (-1, 0, 1))
            for n in range(3):
                new[key[:d] + (n,) + key[d + 1:]] = a * low ** n + b * mid ** n + c * up ** n
        k = new
    K = k
    xx, yy, zz = K[2, 0, 0], K[0, 2, 0], K[0, 0, 2]
    # second order relaxes, every cumulant above it is set to zero
    dxy, dxz, tr = xx - yy, xx - zz, xx + yy + zz
    dxu = -0.5 * w1 * (2.0 * xx - yy - zz) - 0.5 * (tr - 1.0)
    dyv, dzw = dxu + 1.5 * w1 * dxy, dxu + 1.5 * w1 * dxz
    g = 3.0 * (1.0 - 0.5 * w1)
    ux2, uy2, uz2 = (v * v for v in u)
    dxy = (1.0 - w1) * dxy - g * (ux2 * dxu - uy2 * dyv)
    dxz = (1.0 - w1) * dxz - g * (ux2 * dxu - uz2 * dzw)
    tr = 1.0 - 1.5 * (ux2 * dxu + uy2 * dyv + uz2 * dzw)
    xx = (dxy + dxz + tr) / 3.0
    yy, zz = xx - dxy, xx - dxz
    xy, xz, yz = ((1.0 - w1) * K[q] for q in ((1, 1, 0), (1, 0, 1), (0, 1, 1)))
    M = {key: 0.0 for key in K}
    M[0, 0, 0] = 1.0
    M[2, 0, 0], M[0, 2, 0], M[0, 0, 2], M[1, 1, 0], M[1, 0, 1], M[0, 1, 1] = xx, yy, zz, xy, xz, yz
    M[2, 1, 1], M[1, 2, 1], M[1, 1, 2] = xx * yz + 2 * xy * xz, yy * xz + 2 * xy * yz, zz * xy + 2 * xz * yz
    M[2, 2, 0], M[2, 0, 2], M[0, 2, 2] = xx * yy + 2 * xy * xy, xx * zz + 2 * xz * xz, yy * zz + 2 * yz * yz
    s42 = (xx * M[0, 2, 2] + yy * M[2, 0, 2] + zz * M[2, 2, 0]
           + 4.0 * (yz * M[2, 1, 1] + xz * M[1, 2, 1] + xy * M[1, 1, 2]))
    s222 = 8.0 * xy * xz * yz + 2.0 * (xz * xz * yy + yz * yz * xx + xy * xy * zz) + xx * yy * zz
    M[2, 2, 2] = s42 - 2.0 * s222
    # back, axis by axis: the three populations of a line from its moments about u
    k = {key: M[key] * rho for key in M}
    for d in (2, 1, 0):
        v = u[d]
        new = {}
        for key in k:
            if key[d] != 0:
                continue
            m0, m1, m2 = (k[key[:d] + (n,) + key[d + 1:]] for n in range(3))
            r1, r2 = m1 + v * m0, m2 + 2.0 * v * m1 + v * v * m0        # raw moments
            new[key[:d] + (-1,) + key[d + 1:]] = 0.5 * (r2 - r1)
            new[key[:d] + (0,) + key[d + 1:]] = m0 - r2
            new[key[:d] + (1,) + key[d + 1:]] = 0.5 * (r2 + r1)
        k = new
    return torch.stack([k[c] for c in C]), rho, u
