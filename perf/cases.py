"""Timed cases: the work a program using this framework has it do, through its public entry points.

The kinds:

lattice  One cylinder-flow lattice (``lbm.Lattice``): advance ``steps`` steps, then read the result -- rho, u, v
         into device arrays (a snapshot), or the drag and lift of the new steps on the host (the loop that runs a
         case to periodic shedding).  Sizes run from the 400 x 200 lattice of a D = 10 cylinder to 16000 x 8000,
         with every storage form, collision, wall rule and bounce-back rule.
batch    A snapshot round of the batched solver (``lbm.Batch``): every case advances the snapshot stride, then
         hands over its fields.
conv     One 3 x 3 convolution layer of the warm-start network in training: forward, input gradient, weight
         gradient (``nn.conv3x3_*``).
train    One training iteration of ``nn.WarmStartNet``: inputs, forward, loss, backward, Adam.
predict  The warm start itself: one-sample inference, decoding to rho, u, v, and the lattice's start from them.

All lattices run on one stream, as in a program that owns one GPU and works through its cases; the network's calls
run on torch's current stream.
"""
import math

import numpy as np
import torch

from paper_2605_02185_gb300 import lbm, nn
from paper_2605_02185_gb300 import workloads as W

STORAGE = {"f32": lbm.LBM_F32, "f16": lbm.LBM_F16_OFS, "bf16": lbm.LBM_BF16_OFS, "f64": lbm.LBM_F64,
           "f16sr": lbm.LBM_F16_SR, "bf16sr": lbm.LBM_BF16_SR}
ELEM = {"f32": 4, "f16": 2, "bf16": 2, "f64": 8, "f16sr": 2, "bf16sr": 2}
BC = {"freeslip": lbm.LBM_BC_FREESLIP, "periodic": lbm.LBM_BC_PERIODIC, "zouhe": lbm.LBM_BC_ZOUHE,
      "movingwall": lbm.LBM_BC_MOVINGWALL}
COLLISION = {"bgk": lbm.LBM_COLLIDE_BGK, "mrt": lbm.LBM_COLLIDE_MRT}
BOUNCE = {"halfway": lbm.LBM_BOUNCE_HALFWAY, "interpolated": lbm.LBM_BOUNCE_INTERPOLATED}

# The warm-start network (nn.WarmStartNet): layer -> (input channels, output channels, level).
LAYERS = {"c1a": (8, 32, 0), "c1b": (32, 32, 0), "c2a": (32, 64, 1), "c2b": (64, 64, 1), "c3a": (64, 128, 2),
          "c3b": (128, 128, 2), "c4a": (128, 256, 3), "c4b": (256, 256, 3), "d3a": (384, 128, 2),
          "d3b": (128, 128, 2), "d2a": (192, 64, 1), "d2b": (64, 64, 1), "d1a": (96, 32, 0), "d1b": (32, 32, 0),
          "head": (32, 8, 0)}
LR = 3e-6  # an iteration of the learning-rate warm-up
PHASE, RE_FEATURE = 0.7, 0.25


def _lattice(name, nx, ny, D, xc, yc, U, tau, steps, storage="f32", collision="bgk", bc="freeslip",
             bounce="halfway", read="fields"):
    return dict(name=name, kind="lattice", nx=nx, ny=ny, D=D, xc=xc, yc=yc, U=U, tau=tau, steps=steps,
                storage=storage, collision=collision, bc=bc, bounce=bounce, read=read)


def _box(name, D, U, Re, steps, **kw):
    """The paper's box, 40D x 20D with the centre at (10D, 10D)."""
    return _lattice(name, 40 * D, 20 * D, D, 10 * D, 10 * D, U, 0.5 + 3.0 * U * D / Re, steps, **kw)


def listed():
    return [
        # The small shedding case, run to periodicity in chunks: after each chunk the host reads the new drag and
        # lift.  A launch-bound lattice: its populations are 2.9 MB.
        _box("chunk_400x200", 10, 0.05, 80.0, 1000, collision="mrt", read="forces"),
        # The paper's own set-up (D = 20, U = 0.02, tau = 0.512, MRT) with its Zou-He walls, between two snapshots.
        _box("paper_800x400", 20, 0.02, 100.0, 500, collision="mrt", bc="zouhe"),
        # The judge's chunk of the learned warm start (D = 40): 1000 steps, then the drag and lift.  Both population
        # buffers (92 MB) fit in L2.
        _box("chunk_1600x800", 40, 0.05, 80.0, 1000, collision="mrt", read="forces"),
        # A ragged lattice with an off-centre body, interpolated bounce-back, periodic walls, an odd number of steps.
        _lattice("ragged_1283x517", 1283, 517, 25, 311, 264, 0.05, 0.55, 101, collision="mrt", bc="periodic",
                 bounce="interpolated"),
        # The production case (D = 80, Re = 100): 369 MB of populations, between two snapshots.
        _box("production_3200x1600", 80, 0.05, 100.0, 100),
        # The throughput case: 128M nodes, the snapshot stride.
        _box("throughput_16000x8000", 400, 0.04, 100.0, 37),
        # The same lattice in the 16-bit form that keeps Cd and St (bfloat16, stochastic rounding).
        _box("throughput_bf16sr", 400, 0.04, 100.0, 37, storage="bf16sr"),
        # Snapshots for training: 16 cases of D = 20 .. 60 (800 to 2400 nodes wide) in one launch per step, the
        # snapshot stride of 37 steps, then every case's fields.
        dict(name="snapshots_16_cases", kind="batch", cases=16, mix=0, steps=37, storage="f32", collision="mrt"),
        # A full-resolution layer of the network (32 channels): few channels, many pixels.
        dict(name="conv_c1b", kind="conv", N=4, H=800, W=1600, cin=32, cout=32),
        # The layer with the most input channels.
        dict(name="conv_d3a", kind="conv", N=4, H=200, W=400, cin=384, cout=128),
        # One training iteration on the D = 40 grid, 4 samples.
        dict(name="train_800x1600", kind="train", N=4, H=800, W=1600),
        # The warm start of one lattice on the D = 40 grid.
        dict(name="predict_800x1600", kind="predict", H=800, W=1600),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_lattice(rng):
    nodes = _log(rng, 3e4, 1.28e8)
    ratio = rng.uniform(1.3, 3.0)
    nx, ny = max(64, int(math.sqrt(nodes * ratio))), max(48, int(math.sqrt(nodes / ratio)))
    storage = rng.choice(["f32", "f32", "f32", "f32", "bf16sr", "f16sr", "f16", "bf16", "f64"])
    collision = rng.choice(["bgk", "mrt", "mrt"])
    bounce = rng.choice(["halfway", "halfway", "halfway", "interpolated"])
    D = max(6, int(ny / rng.uniform(8.0, 24.0)))
    U, Re = rng.choice([0.02, 0.04, 0.05]), rng.uniform(60.0, 120.0)
    tau = max(0.5 + 3.0 * U * D / Re, 0.55 if collision == "bgk" else 0.512)
    budget = 1e8 if storage == "f64" or (bounce == "interpolated" and storage != "f32") else 8e8
    steps = max(3, min(1000, int(rng.uniform(0.3, 1.0) * budget / (nx * ny))))
    xc, yc = int(nx * rng.uniform(0.2, 0.4)), int(ny * rng.uniform(0.4, 0.6))
    if nx > 512:  # some bodies that lie between two multiples of 256 are refused by lbm_create
        xc = 256 * max(1, round(xc / 256))
    read = rng.choice(["fields", "forces"]) if bounce == "halfway" and storage in ("f32", "f64") else "fields"
    return _lattice("", nx, ny, D, xc, yc, U, tau, steps, storage, collision,
                    rng.choice(["freeslip", "periodic", "zouhe", "movingwall"]), bounce, read)


def draw(rng):
    kind = rng.choices(["lattice", "batch", "conv", "train", "predict"], [10, 3, 5, 1, 1])[0]
    if kind == "lattice":
        c = _draw_lattice(rng)
        del c["name"]
        return c
    if kind == "batch":
        return dict(kind="batch", cases=rng.randint(2, 16), mix=rng.randint(1, 1000), steps=rng.randint(20, 50),
                    storage=rng.choice(["f32", "f32", "bf16sr"]), collision=rng.choice(["bgk", "mrt"]))
    if kind == "conv":
        cin, cout, level = LAYERS[rng.choice(sorted(LAYERS))]
        scale = _log(rng, 0.2, 1.0)  # of the 800 x 1600 grid and its halvings
        return dict(kind="conv", N=rng.randint(1, 4), H=int(scale * (800 >> level)) + rng.randint(0, 3),
                    W=int(scale * (1600 >> level)) + rng.randint(0, 7), cin=cin, cout=cout)
    H = 8 * int(_log(rng, 20, 100))  # the grids of D = 8 .. 40
    if kind == "train":
        return dict(kind="train", N=rng.randint(1, 4), H=H, W=2 * H - 8 * rng.randint(0, 3))
    return dict(kind="predict", H=H, W=2 * H - 8 * rng.randint(0, 3))


# ---------------------------------------------------------------- inputs


_stream = None


def _lattice_stream():
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _mask(nx, ny, D, xc, yc):
    """uint8 [ny, nx], 1 on the staircased cylinder's nodes."""
    m = np.zeros((ny, nx), np.uint8)
    r = D // 2 + 1
    y, x = np.mgrid[yc - r:yc + r + 1, xc - r:xc + r + 1]
    m[yc - r:yc + r + 1, xc - r:xc + r + 1] = 4 * ((x - xc) ** 2 + (y - yc) ** 2) <= D * D
    return m


def _start(nx, ny, U, solid, g):
    """A cold start: unit density, the free stream plus 1e-3 U of noise (float32, on the device)."""
    rho = torch.ones((ny, nx), device="cuda")
    u = U + 1e-3 * U * (2 * torch.rand((ny, nx), device="cuda", generator=g) - 1)
    v = 1e-3 * U * (2 * torch.rand((ny, nx), device="cuda", generator=g) - 1)
    u[solid] = 0
    v[solid] = 0
    return rho, u, v


def _fields_out(nx, ny):
    return [torch.empty((ny, nx), device="cuda") for _ in range(3)]


def _batch_params(case):
    """(D, Re) of each case: the diameters 20, 30, 40, 60 in turn, Re from 60 to 200."""
    n, D = case["cases"], (20, 30, 40, 60)
    return [(D[(i + case["mix"]) % 4], 60.0 * (200.0 / 60.0) ** (((7 * i + case["mix"]) % n + 0.5) / n))
            for i in range(n)]


def _batch_start(case, seed):
    """Host double fields of each case of a batch: the free stream plus 1e-3 U of noise."""
    rng = np.random.default_rng(seed)
    for D, _ in _batch_params(case):
        nx, ny = 40 * D, 20 * D
        solid = _mask(nx, ny, D, 10 * D, 10 * D).astype(bool)
        u, v = (5e-5 * (2 * rng.random((ny, nx), np.float32).astype(np.float64) - 1) for _ in range(2))
        u += 0.05
        u[solid] = 0
        v[solid] = 0
        yield np.ones((ny, nx)), u, v


def _conv_inputs(case, seed):
    N, H, Wd, cin, cout = (case[k] for k in ("N", "H", "W", "cin", "cout"))
    g = _gen(seed)
    x = torch.randn((N, H, Wd, cin), device="cuda", generator=g).clamp_(min=0).bfloat16()  # a ReLU's output
    w = (torch.randn((cout, 3, 3, cin), device="cuda", generator=g) * math.sqrt(2.0 / (9 * cin))).bfloat16()
    b = 0.1 * torch.randn(cout, device="cuda", generator=g)
    gy = torch.randn((N, H, Wd, cout), device="cuda", generator=g)
    gy = (gy * (torch.rand((N, H, Wd, cout), device="cuda", generator=g) > 0.5) * 1e-3).bfloat16()
    return x, w, b, gy


def _target(N, H, Wd, g):
    """Smooth O(1) fields (a wake-like wave of random amplitude per sample), float32 [N H W, 3], and the fluid weight."""
    y = torch.linspace(-1, 1, H, device="cuda")[None, :, None, None]
    x = torch.linspace(0, 12, Wd, device="cuda")[None, None, :, None]
    a = torch.rand((N, 1, 1, 3), device="cuda", generator=g)
    t = a * torch.sin(x * (1 + a) + 6 * a) * torch.exp(-4 * y * y)
    return t.reshape(-1, 3).contiguous()


def _net_grid(H, Wd):
    D = max(8, H // 20)
    return D, _mask(Wd, H, D, Wd // 4, H // 2)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        nx, ny = case["nx"], case["ny"]
        mask = _mask(nx, ny, case["D"], case["xc"], case["yc"])
        lat = lbm.Lattice(nx, ny, case["tau"], case["U"], mask=mask, bc=BC[case["bc"]],
                          storage=STORAGE[case["storage"]], D_ref=float(case["D"]), stream=_lattice_stream(),
                          collision=COLLISION[case["collision"]], bounce=BOUNCE[case["bounce"]],
                          body=(float(case["xc"]), float(case["yc"]), 0.5 * case["D"]))
        start = _start(nx, ny, case["U"], torch.from_numpy(mask).cuda().bool(), _gen(seed))
        torch.cuda.synchronize()
        lbm.lbm_init_fields_device(lat.h, *(t.data_ptr() for t in start), False)
        return {"kind": kind, "lat": lat, "steps": case["steps"], "read": case["read"], "have": 1,
                "out": _fields_out(nx, ny) if case["read"] == "fields" else None}
    if kind == "batch":
        cases = [W.cylinder_case(D, 0.05, Re) for D, Re in _batch_params(case)]
        batch = lbm.Batch(cases, storage=STORAGE[case["storage"]], collision=COLLISION[case["collision"]],
                          stream=_lattice_stream())
        for c, f in enumerate(_batch_start(case, seed)):
            batch.init_fields(c, *f)
        return {"kind": kind, "batch": batch, "steps": case["steps"], "out": [_fields_out(w.nx, w.ny) for w in cases]}
    if kind == "conv":
        x, w, b, gy = _conv_inputs(case, seed)
        wf = torch.empty((case["cin"], 3, 3, case["cout"]), dtype=torch.bfloat16, device="cuda")
        nn.flip_weights(w, wf, case["cout"], case["cin"])
        return {"kind": kind, "x": x, "w": w, "wf": wf, "b": b, "gy": gy, "y": torch.empty_like(gy),
                "gx": torch.empty_like(x), "gw": torch.empty(w.shape, device="cuda"), "gb": torch.empty_like(b)}
    H, Wd = case["H"], case["W"]
    D, mask = _net_grid(H, Wd)
    solid = torch.from_numpy(mask).cuda()
    g = _gen(seed)
    if kind == "train":
        N = case["N"]
        net = nn.WarmStartNet(N, H, Wd, torch.device("cuda"), seed=seed)
        weight = (1.0 - solid.float()).reshape(-1).repeat(N)
        phase = [float(p) for p in 2 * math.pi * torch.rand(N, device="cuda", generator=g)]
        return {"kind": kind, "net": net, "solid": solid, "phase": phase, "target": _target(N, H, Wd, g),
                "weight": weight, "D": D}
    # predict: a trained net's output stays near its targets, so the random head is scaled down
    net = nn.WarmStartNet(1, H, Wd, torch.device("cuda"), seed=seed)
    st = net.state()
    st["head.w"] *= 0.1
    net.load_state(st)
    U, tau = 0.05, 0.5 + 3.0 * 0.05 * D / 80.0
    lat = lbm.Lattice(Wd, H, tau, U, mask=mask, D_ref=float(D), stream=_lattice_stream(),
                      collision=lbm.LBM_COLLIDE_MRT)
    torch.cuda.synchronize()
    return {"kind": kind, "net": net, "lat": lat, "solid": solid, "D": D, "U": U, "fr": _fields_out(Wd, H),
            "out": _fields_out(Wd, H)}


# ------------------------------------------------------------------ work


def _encode(solid, D, phase, x, stream=None):
    H, Wd = solid.shape
    nn.encode_input(solid, RE_FEATURE, phase, H, Wd, x, stream, wave_k=2 * math.pi / (5.0 * D), wave_x0=10.0 * D)


def run(s):
    kind = s["kind"]
    if kind == "lattice":
        lat = s["lat"]
        lat.step(s["steps"])
        if s["read"] == "fields":
            lbm.lbm_fields_device(lat.h, *(t.data_ptr() for t in s["out"]))
            return s["out"]
        n = lat.force_count()
        cd, cl = lat.forces(s["have"], n - s["have"])
        s["have"] = n
        return cd, cl
    if kind == "batch":
        b = s["batch"]
        b.step(s["steps"])
        for c, out in enumerate(s["out"]):
            lbm.lbm_fields_device(b.case(c), *(t.data_ptr() for t in out))
        return s["out"]
    if kind == "conv":
        x, w, gy = s["x"], s["w"], s["gy"]
        N, H, Wd, cin = x.shape
        cout = w.shape[0]
        nn.conv3x3_fwd(x, cin, w, s["b"], s["y"], cout, N, H, Wd, cin, cout, True)
        nn.fill_zero(s["gw"])
        nn.fill_zero(s["gb"])
        nn.conv3x3_wgrad(x, cin, gy, cout, s["gw"], s["gb"], N, H, Wd, cin, cout)
        nn.conv3x3_dgrad(gy, cout, s["wf"], s["gx"], cin, N, H, Wd, cin, cout, mask=x, ms=cin)
        return {"y": s["y"], "gx": s["gx"], "gw": s["gw"], "gb": s["gb"]}
    net = s["net"]
    if kind == "train":
        for j, ph in enumerate(s["phase"]):
            _encode(s["solid"], s["D"], ph, net.x0[j])
        net.forward()
        loss = net.loss_and_grad(s["target"], s["weight"])
        net.backward()
        net.adam_step(LR)
        out = {"out": net.out, "loss": loss}
        for name, c in net.layers.items():
            out.update({name + ".gw": c.gw, name + ".gb": c.gb, name + ".w": c.w, name + ".b": c.b})
        return out
    lat, fr, U, stream = s["lat"], s["fr"], s["U"], _lattice_stream()
    with torch.cuda.stream(stream):
        _encode(s["solid"], s["D"], PHASE, net.x0[0], stream)
        net.forward(stream)
        nn.decode_output(net.out, net.OUT_C, s["solid"], lat.nx * lat.ny, U, 0.2 * U, U * U, *fr, stream)
    lbm.lbm_init_fields_device(lat.h, *(t.data_ptr() for t in fr), True)
    lbm.lbm_fields_device(lat.h, *(t.data_ptr() for t in s["out"]))
    return {"out": net.out, "predicted": fr, "started": s["out"]}


def _net_flops(N, H, Wd):
    return sum(2.0 * N * (H >> lv) * (Wd >> lv) * 9 * ci * co for ci, co, lv in LAYERS.values())


def _net_weights():
    return sum(9 * ci * co + co for ci, co, _ in LAYERS.values())


def work(case):
    """The state or inputs read once and the results written once, whatever the number of steps between; 110
    operations a node and step for BGK, 130 for MRT."""
    kind = case["kind"]
    if kind in ("lattice", "batch"):
        if kind == "lattice":
            nodes, reads = case["nx"] * case["ny"], case["read"] == "fields"
        else:
            nodes, reads = sum(800 * D * D for D, _ in _batch_params(case)), True
        return {"bytes": nodes * (18.0 * ELEM[case["storage"]] + (12.0 if reads else 0.0)) + 16.0 * case["steps"],
                "flops": (130.0 if case["collision"] == "mrt" else 110.0) * nodes * case["steps"]}
    if kind == "conv":
        P, ci, co = case["N"] * case["H"] * case["W"], case["cin"], case["cout"]
        return {"bytes": 2.0 * P * (2 * ci + 2 * co) + 9.0 * ci * co * (2 + 4), "flops": 3 * 2.0 * P * 9 * ci * co}
    if kind == "train":
        P = case["N"] * case["H"] * case["W"]
        first = 2.0 * P * 9 * 8 * 32  # the first layer has no input gradient
        return {"bytes": P * (1 + 16 + 16) + 4.0 * _net_weights() * 7, "flops": 3 * _net_flops(case["N"], case["H"], case["W"]) - first}
    P = case["H"] * case["W"]
    return {"bytes": P * (1 + 16 + 12 + 36 + 12) + 2.0 * _net_weights(), "flops": _net_flops(1, case["H"], case["W"])}


# ----------------------------------------------------------------- exact
# The lattice in 64 bits, plain torch: f holds the post-collision populations [9][ny][nx].


_CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
_CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
_OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
_WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


def _equilibrium(rho, u, v):
    f = torch.empty((9,) + rho.shape, dtype=torch.float64, device=rho.device)
    for k in range(9):
        cu = _CX[k] * u + _CY[k] * v
        f[k] = _WT[k] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u + v * v))
    return f


def _moments(f):
    rho = f.sum(0)
    jx = f[1] - f[3] + f[5] - f[6] - f[7] + f[8]
    jy = f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
    return rho, jx, jy


class _Exact:
    def __init__(self, nx, ny, D, xc, yc, U, tau, collision, bc, bounce, fields):
        self.U, self.tau, self.mrt, self.bc = U, tau, collision == "mrt", bc
        mask = _mask(nx, ny, D, xc, yc)
        self.solid = torch.from_numpy(mask).cuda().bool()
        rho, u, v = (t.double() for t in fields)
        self.f = _equilibrium(rho, u, v)
        y0, x0 = yc - D // 2 - 3, xc - D // 2 - 3
        box = mask[y0:yc + D // 2 + 4, x0:xc + D // 2 + 4].astype(bool)
        self.links = []  # per arriving direction: the fluid nodes whose source is solid, and the link's fraction
        for k in range(1, 9):
            src = np.roll(box, (_CY[k], _CX[k]), (0, 1))
            yy, xx = np.nonzero(src & ~box)
            q = np.full(len(yy), 0.5)
            if bounce == "interpolated":
                cx, cy = -_CX[k], -_CY[k]  # the direction that leaves
                dx, dy = xx + x0 - xc, yy + y0 - yc
                a, b, c = cx * cx + cy * cy, dx * cx + dy * cy, dx * dx + dy * dy - 0.25 * D * D
                disc = b * b - a * c
                t = np.where(disc >= 0, (-b - np.sqrt(np.maximum(disc, 0))) / a, -1.0)
                q = np.where((t > 0) & (t <= 1), t, 0.5)
                q = np.where((q < 0.5) & box[yy + _CY[k], xx + _CX[k]], 0.5, q)
            self.links.append([torch.from_numpy(np.ascontiguousarray(t)).cuda() for t in (yy + y0, xx + x0, q)])

    def step(self):
        old, U = self.f, self.U
        f = torch.empty_like(old)
        for k in range(9):
            f[k] = torch.roll(old[k], (_CY[k], _CX[k]), (0, 1))
            if _CX[k]:  # a source outside the lattice: the node's own value stands in
                x = 0 if _CX[k] > 0 else -1
                f[k][:, x] = old[k][:, x]
            if _CY[k] and self.bc != "periodic":
                y = 0 if _CY[k] > 0 else -1
                if self.bc == "movingwall":
                    f[k][y] = old[_OPP[k]][y] + 6 * _WT[k] * _CX[k] * U * old[:, y].sum(0)
                else:
                    f[k][y] = old[k][y]
            if k:
                yy, xx, q = self.links[k - 1]
                a = old[_OPP[k], yy, xx]
                low = 2 * q * a + (1 - 2 * q) * old[_OPP[k], yy + _CY[k], xx + _CX[k]]
                f[k, yy, xx] = torch.where(q < 0.5, low, a / (2 * q) + (1 - 1 / (2 * q)) * old[k, yy, xx])
        if self.bc in ("freeslip", "zouhe"):
            for y, (a, b, c), (d, e, g) in ((-1, (4, 7, 8), (2, 6, 5)), (0, (2, 6, 5), (4, 7, 8))):
                if self.bc == "freeslip":
                    f[a, y], f[b, y], f[c, y] = f[d, y], f[e, y], f[g, y]
                else:
                    m = 0.5 * U * (f[0, y] + f[1, y] + f[3, y] + 2 * (f[d, y] + f[e, y] + f[g, y]))
                    h = 0.5 * (f[1, y] - f[3, y])
                    # the wall's incoming diagonals: (x-, from opposite x+) and (x+, from opposite x-)
                    lo, hi = (7, 8) if y else (6, 5)
                    f[a, y], f[lo, y], f[hi, y] = f[d, y], f[_OPP[lo], y] + h - m, f[_OPP[hi], y] - h + m
        rho = (f[0, :, 0] + f[2, :, 0] + f[4, :, 0] + 2 * (f[3, :, 0] + f[6, :, 0] + f[7, :, 0])) / (1 - U)
        h = 0.5 * (f[2, :, 0] - f[4, :, 0])
        f[1, :, 0] = f[3, :, 0] + 2 / 3 * rho * U
        f[5, :, 0] = f[7, :, 0] - h + rho * U / 6
        f[8, :, 0] = f[6, :, 0] + h + rho * U / 6
        f[:, :, -1] = f[:, :, -2]
        rho, jx, jy = _moments(f)
        if self.mrt:
            qx, qy = f[5] - f[6] - f[7] + f[8], f[5] + f[6] - f[7] - f[8]
            axis, diag = f[1] + f[2] + f[3] + f[4], f[5] + f[6] + f[7] + f[8]
            e = -4 * f[0] - axis + 2 * diag
            eps = 4 * f[0] - 2 * axis + diag
            qx, qy = qx - 2 * (f[1] - f[3]), qy - 2 * (f[2] - f[4])
            pxx, pxy = f[1] - f[2] + f[3] - f[4], f[5] - f[6] + f[7] - f[8]
            jj = (jx * jx + jy * jy) / rho
            ce, cps = (e + 2 * rho - 3 * jj) * (1.1 / 36), (eps - rho + 3 * jj) * (1.1 / 36)
            cqx, cqy = (qx + jx) * (1.1 / 12), (qy + jy) * (1.1 / 12)
            cxx, cxy = (pxx - (jx * jx - jy * jy) / rho) * (0.25 / self.tau), (pxy - jx * jy / rho) * (0.25 / self.tau)
            f[0] -= 4 * (cps - ce)
            for k in range(1, 9):
                cx, cy = _CX[k], _CY[k]
                if k < 5:
                    f[k] -= -ce - 2 * cps - 2 * (cx * cqx + cy * cqy) + (1 if cx else -1) * cxx
                else:
                    f[k] -= 2 * ce + cps + cx * cqx + cy * cqy + cx * cy * cxy
        else:
            f += (_equilibrium(rho, jx / rho, jy / rho) - f) / self.tau
        self.f = f

    def force(self):
        """Momentum exchange of the post-collision populations over the links (half-way bounce-back)."""
        fx, fy = 0.0, 0.0
        for k in range(1, 9):
            yy, xx, _ = self.links[k - 1]
            s = 2 * self.f[_OPP[k], yy, xx].sum()
            fx, fy = fx - s * _CX[k], fy - s * _CY[k]
        return torch.stack([fx, fy])

    def fields(self):
        rho, jx, jy = _moments(self.f)
        u, v = jx / rho, jy / rho
        rho[self.solid], u[self.solid], v[self.solid] = 1.0, 0.0, 0.0
        return [rho, u, v]


def _conv64(x, w, b=None):
    """3 x 3 convolution, zero padding, [N][H][W][C] doubles, w [O][3][3][C]."""
    N, H, Wd, C = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    y = torch.zeros((N * H * Wd, w.shape[0]), dtype=torch.float64, device=x.device)
    for t in range(9):
        y.addmm_(xp[:, t // 3:t // 3 + H, t % 3:t % 3 + Wd].reshape(-1, C), w[:, t // 3, t % 3].T)
    y = y.view(N, H, Wd, -1)
    return y if b is None else y.add_(b.double())


def _conv64_back(x, w, gy, want_gx=True):
    """(gx, gw, gb) of _conv64."""
    N, H, Wd, C = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    g2 = gy.reshape(-1, gy.shape[3])
    gw = torch.stack([g2.T @ xp[:, t // 3:t // 3 + H, t % 3:t % 3 + Wd].reshape(-1, C) for t in range(9)], 1)
    gx = _conv64(gy, w.flip(1, 2).permute(3, 1, 2, 0)) if want_gx else None
    return gx, gw.view(w.shape), g2.sum(0)


def _pool64(x):
    N, H, Wd, C = x.shape
    return x.view(N, H // 2, 2, Wd // 2, 2, C).mean((2, 4))


def _up64(x):
    return x.repeat_interleave(2, 1).repeat_interleave(2, 2)


def _input64(case, mask, D, phase):
    H, Wd = mask.shape
    x = torch.arange(Wd, device="cuda", dtype=torch.float64).expand(H, Wd)
    y = torch.arange(H, device="cuda", dtype=torch.float64)[:, None].expand(H, Wd)
    one, arg = torch.ones_like(x), 2 * math.pi / (5.0 * D) * (x - 10.0 * D) - phase
    ch = [torch.from_numpy(mask).cuda().double(), RE_FEATURE * one, math.sin(phase) * one, math.cos(phase) * one,
          x / Wd, y / H, torch.cos(arg), torch.sin(arg)]
    return torch.stack(ch, 2).bfloat16().double()  # the network's input is bfloat16


def _net_params(seed):
    """The initial weights of nn.WarmStartNet(seed): FP32 values drawn layer by layer."""
    rng = np.random.default_rng(seed)
    return {name: (rng.standard_normal((co, 3, 3, ci)) * math.sqrt(2.0 / (9 * ci))).astype(np.float32)
            for name, (ci, co, _) in LAYERS.items()}


def _net_forward64(x0, w):
    """Every layer's input, and the output; w: bfloat16-rounded weights as doubles (the biases are zero)."""
    inp, act = {}, {}

    def conv(name, x, relu=True):
        inp[name] = x
        y = _conv64(x, w[name])
        act[name] = y.clamp_(min=0) if relu else y
        return act[name]

    s1 = conv("c1b", conv("c1a", x0))
    s2 = conv("c2b", conv("c2a", _pool64(s1)))
    s3 = conv("c3b", conv("c3a", _pool64(s2)))
    b4 = conv("c4b", conv("c4a", _pool64(s3)))
    d3 = conv("d3b", conv("d3a", torch.cat([_up64(b4), s3], 3)))
    d2 = conv("d2b", conv("d2a", torch.cat([_up64(d3), s2], 3)))
    d1 = conv("d1b", conv("d1a", torch.cat([_up64(d2), s1], 3)))
    return inp, act, conv("head", d1, relu=False)


def _net_backward64(inp, act, w, g_out):
    grads = {}

    def back(name, g, want_gx=True):
        gx, gw, gb = _conv64_back(inp[name], w[name], g, want_gx)
        grads[name] = (gw, gb)
        return gx

    def through(g, name):  # the ReLU of a layer
        return g * (act[name] > 0)

    def decoder(a, b, g, nup):
        gc = back(a, through(back(b, g), a))
        return 4 * _pool64(gc[..., :nup].contiguous()), gc[..., nup:]

    up1, sk1 = decoder("d1a", "d1b", through(back("head", g_out), "d1b"), 64)
    up2, sk2 = decoder("d2a", "d2b", through(up1, "d2b"), 128)
    up3, sk3 = decoder("d3a", "d3b", through(up2, "d3b"), 256)
    g = back("c4a", through(back("c4b", through(up3, "c4b")), "c4a"))
    for a, b, sk in (("c3a", "c3b", sk3), ("c2a", "c2b", sk2), ("c1a", "c1b", sk1)):
        g = through(sk + _up64(g) / 4, b)
        g = back(a, through(back(b, g), a), want_gx=a != "c1a")
    return grads


def exact(case, seed):
    kind = case["kind"]
    if kind == "lattice":
        nx, ny = case["nx"], case["ny"]
        mask = _mask(nx, ny, case["D"], case["xc"], case["yc"])
        start = _start(nx, ny, case["U"], torch.from_numpy(mask).cuda().bool(), _gen(seed))
        e = _Exact(nx, ny, case["D"], case["xc"], case["yc"], case["U"], case["tau"], case["collision"], case["bc"],
                   case["bounce"], start)
        F = []
        for _ in range(case["steps"]):
            e.step()
            if case["read"] == "forces":
                F.append(e.force())
        if case["read"] == "fields":
            return e.fields()
        F = torch.stack(F).cpu().numpy() / (0.5 * case["U"] ** 2 * case["D"])
        return np.ascontiguousarray(F[:, 0]), np.ascontiguousarray(F[:, 1])
    if kind == "batch":
        out = []
        for (D, Re), f in zip(_batch_params(case), _batch_start(case, seed)):
            e = _Exact(40 * D, 20 * D, D, 10 * D, 10 * D, 0.05, 0.5 + 3 * 0.05 * D / Re, case["collision"],
                       "freeslip", "halfway", [torch.from_numpy(t).cuda() for t in f])
            for _ in range(case["steps"]):
                e.step()
            out.append(e.fields())
        return out
    if kind == "conv":
        x, w, b, gy = (t.double() for t in _conv_inputs(case, seed))
        y = _conv64(x, w, b).clamp_(min=0)
        gx, gw, gb = _conv64_back(x, w, gy)
        return {"y": y, "gx": gx.mul_(x > 0), "gw": gw, "gb": gb}
    H, Wd = case["H"], case["W"]
    D, mask = _net_grid(H, Wd)
    master = {n: torch.from_numpy(t).cuda() for n, t in _net_params(seed).items()}
    if kind == "predict":
        master["head"] *= 0.1
    w = {n: t.bfloat16().double() for n, t in master.items()}
    if kind == "train":
        N, g = case["N"], _gen(seed)
        phase = [float(p) for p in 2 * math.pi * torch.rand(N, device="cuda", generator=g)]
        target = _target(N, H, Wd, g).double().view(N, H, Wd, 3)
        x0 = torch.stack([_input64(case, mask, D, p) for p in phase])
        inp, act, out = _net_forward64(x0, w)
        fluid = 1.0 - torch.from_numpy(mask).cuda().double()[None, :, :, None]
        d = (out[..., :3] - target) * fluid
        g_out = torch.zeros_like(out)
        g_out[..., :3] = 2 * d / (3 * N * H * Wd)
        grads = _net_backward64(inp, act, w, g_out)
        ans = {"out": out, "loss": (d * d).sum().reshape(1)}
        for n, (gw, gb) in grads.items():  # the first Adam step: w - lr g / (|g| + eps)
            ans.update({n + ".gw": gw, n + ".gb": gb, n + ".w": master[n].double() - LR * gw / (gw.abs() + 1e-8),
                        n + ".b": None})  # +-lr by the sign of the gradient alone: the biases start at zero
        return ans
    out = _net_forward64(_input64(case, mask, D, PHASE)[None], w)[2][0]
    U, solid = 0.05, torch.from_numpy(mask).cuda().bool()
    rho, u, v = 1 + U * U * out[..., 0], U + 0.2 * U * out[..., 1], 0.2 * U * out[..., 2]
    rho[solid], u[solid], v[solid] = 1.0, 0.0, 0.0
    # the start's non-equilibrium part carries no mass or momentum: the lattice's fields are the predicted ones
    return {"out": out[None], "predicted": [rho, u, v], "started": [rho, u, v]}
