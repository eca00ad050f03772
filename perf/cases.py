"""Performance cases of the library: what its users have it do, through the public entry points.

Every case is a dict of plain values.  `prepare` makes what a user's program holds before the call (the geometry, the
context with its boundary conditions and start state, the device buffers), `run` is one pass of that program, `work`
the bytes and operations the pass cannot do without, `exact` the same outputs in 64 bits from plain torch.

Kinds:
  flow      one lattice: a 100-step (or shorter) stretch of a run and the fields after it (Lattice)
  ensemble  a batched ensemble of packs, cold start to the fields of every member (Batch)
  colour    the two-fluid model with a non-wetting fluid injected, and its fields (ColorLattice)
  conv      one 3x3x3 convolution layer of the warm-start network on device buffers (conv3d_bf16)
  grad      loss and gradient of the warm-start network, one training batch (WarmStartNet.loss_grad)
  predict   inference of the warm-start network on one geometry (WarmStartNet.predict)

Sizes are the repository's: the 16x16x64 duct and the 256^3 sphere pack (radii 6-12, porosity 0.35, six reservoir
layers) of the flow benchmark, packs with edges 64..160 of the ensemble, 64^3 training volumes in batches of 8, the
radii 5-10 pack of the two-fluid run; others are ragged volumes between them.
"""
import math

import numpy as np
import torch

from paper_1806_10589_gb300 import Batch, ColorLattice, Lattice, WarmStartNet, conv3d_bf16

# D3Q19 in the library's order (opposites are (odd q, q + 1)) and its weights
XI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
BYTES = {"fp64": 8, "fp32": 4, "fp16dev": 2, "bf16dev": 2}


def listed():
    return [
        # The 16x16x64 duct in FP64: the validation problem, the smallest call a user makes (launch latency), one
        # check interval of the convergence loop with its flux samples.
        dict(name="duct_fp64", kind="flow", geometry="duct", nx=16, ny=16, nz=64, tau=1.0, precision="fp64", variant=0,
             steps=100, sample=True),
        # A small ragged sample, default kernel, FP32: the same convergence loop on a core-plug sub-volume.
        dict(name="small_fp32", kind="flow", geometry="pack", nx=61, ny=67, nz=72, tau=0.7, precision="fp32", variant=0,
             steps=100, sample=True),
        # The benchmark's lattice: 256^3 pack, FP32, AA pattern; a stretch of the long run to steady flux.
        dict(name="pack256_fp32", kind="flow", geometry="pack", nx=256, ny=256, nz=256, tau=0.7, precision="fp32",
             variant=3, steps=100, sample=False),
        # The largest storage-reduced run: a ragged pack of about 256^3 in FP16 deviations, AA pattern.
        dict(name="pack251_fp16", kind="flow", geometry="pack", nx=251, ny=243, nz=262, tau=0.7, precision="fp16dev",
             variant=3, steps=100, sample=False),
        # A mid-size ragged pack in BF16 deviations on the library's default kernel.
        dict(name="pack157_bf16", kind="flow", geometry="pack", nx=157, ny=149, nz=171, tau=0.8, precision="bf16dev",
             variant=0, steps=100, sample=False),
        # An FP64 reference run of a pack (the state every other storage format is judged against).
        dict(name="pack125_fp64", kind="flow", geometry="pack", nx=128, ny=121, nz=135, tau=0.7, precision="fp64",
             variant=0, steps=50, sample=False),
        # The ensemble: packs of uneven size from rest in one batch, FP16 deviations, then every member's fields
        # (the training data of the warm start).
        dict(name="ensemble6_fp16", kind="ensemble", members=6, lo=64, hi=160, tau=0.7, precision="fp16dev", steps=1200),
        # Drainage: the two-fluid colour model in FP32, one output interval of the 50,000-step run.
        dict(name="colour_fp32", kind="colour", nx=128, ny=128, nz=256, tau=0.7, precision="fp32", steps=1000),
        # The network's most frequent layer, forward, on a training batch.
        dict(name="conv_fwd_32", kind="conv", op=0, batch=8, nx=64, ny=64, nz=64, cin=32, cout=32),
        # A weight gradient at a ragged volume.
        dict(name="conv_wgrad_64", kind="conv", op=2, batch=4, nx=44, ny=52, nz=36, cin=64, cout=64),
        # A training step's loss and gradient: the specified network, a batch of 64^3 crops.
        dict(name="grad_8x64", kind="grad", batch=8, nx=64, ny=64, nz=64, levels=4, base=32),
        # Inference on a new geometry: the warm start of a ragged volume.
        dict(name="predict_128", kind="predict", nx=128, ny=120, nz=136, levels=4, base=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flow", "flow", "flow", "ensemble", "colour", "conv", "conv", "grad", "predict"])
    if kind == "flow":
        prec = rng.choice(["fp64", "fp32", "fp16dev", "bf16dev"])
        hi = 150 if prec == "fp64" else 250
        d = [_log(rng, 16, hi) for _ in range(3)]
        return dict(kind=kind, geometry="duct" if max(d) < 48 else "pack", nx=d[0], ny=d[1], nz=max(24, d[2]),
                    tau=rng.choice([0.7, 0.8, 1.0]), precision=prec, variant=rng.choice([0, 3]),
                    steps=rng.choice([20, 50, 100]), sample=rng.random() < 0.5)
    if kind == "ensemble":
        lo = _log(rng, 24, 80)
        return dict(kind=kind, members=rng.randint(3, 6), lo=lo, hi=rng.randint(lo + 1, 2 * lo), tau=0.7,
                    precision=rng.choice(["fp16dev", "fp32", "bf16dev"]), steps=rng.randint(200, 1200))
    if kind == "colour":
        return dict(kind=kind, nx=_log(rng, 20, 120), ny=_log(rng, 20, 120), nz=_log(rng, 40, 200), tau=0.7,
                    precision=rng.choice(["fp32", "fp32", "fp64"]), steps=rng.randint(100, 300))
    if kind == "conv":
        c = [32, 64, 128, 256]
        k = rng.randrange(4)
        side = [72, 48, 24, 12][k]
        return dict(kind=kind, op=rng.randrange(3), batch=rng.randint(1, 8), nx=_log(rng, 6, side), ny=_log(rng, 6, side),
                    nz=_log(rng, 6, side), cin=c[max(0, k - rng.randrange(2))], cout=c[k])
    if kind == "grad":
        return dict(kind=kind, batch=rng.randint(1, 8), nx=8 * rng.randint(2, 8), ny=8 * rng.randint(2, 8),
                    nz=8 * rng.randint(2, 8), levels=rng.choice([3, 4]), base=32)
    return dict(kind=kind, nx=8 * rng.randint(4, 18), ny=8 * rng.randint(4, 16), nz=8 * rng.randint(4, 18),
                levels=rng.choice([3, 4]), base=32)


# ------------------------------------------------------------------ inputs ---
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _pack(nx, ny, nz, seed, porosity=0.35, rmin=6.0, rmax=12.0, reservoir=6):
    """uint8 [z][y][x] mask (1 = solid) of randomly placed spheres that may overlap, on the GPU; `reservoir` clear
    layers at both z ends.  The number of spheres follows from the porosity (Poisson: phi = exp(-n V / box))."""
    g = _gen(seed)
    mean_v = 4 / 3 * math.pi * (rmax ** 4 - rmin ** 4) / (4 * (rmax - rmin))
    m = int(math.ceil(rmax))
    lo = torch.tensor([-m, -m, -m], device="cuda")
    box = torch.tensor([nz, ny, nx], device="cuda")
    n = max(1, int(round(-math.log(porosity) * float((nx + 2 * m) * (ny + 2 * m) * (nz + 2 * m)) / mean_v)))
    c = torch.rand(n, 3, generator=g, device="cuda") * (box + 2 * m) + lo
    r = rmin + (rmax - rmin) * torch.rand(n, generator=g, device="cuda")
    k = torch.arange(-m, m + 1, device="cuda")
    st = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    mask = torch.zeros(nz * ny * nx + 1, dtype=torch.uint8, device="cuda")
    for a in range(0, n, 512):
        ci = c[a:a + 512].floor()
        v = ci[:, None, :].long() + st[None]
        inside = ((v + 0.5 - c[a:a + 512, None, :]).square().sum(-1) <= r[a:a + 512, None].square())
        inside &= ((v >= 0) & (v < box)).all(-1)
        flat = (v[..., 0] * ny + v[..., 1]) * nx + v[..., 2]
        mask[torch.where(inside, flat, nz * ny * nx)] = 1
    mask = mask[:-1].reshape(nz, ny, nx)
    res = min(reservoir, (nz - 1) // 3)
    if res:
        mask[:res] = 0
        mask[nz - res:] = 0
    return mask


def _duct(nx, ny, nz):
    mask = torch.ones(nz, ny, nx, dtype=torch.uint8, device="cuda")
    mask[:, 1:ny - 1, 1:nx - 1] = 0
    return mask


def _flow_mask(case, seed):
    if case["geometry"] == "duct":
        return _duct(case["nx"], case["ny"], case["nz"])
    return _pack(case["nx"], case["ny"], case["nz"], seed)


def _flow_start(case, mask, seed):
    """(Q, rho, u) of a run that is under way: a pressure ramp along z of the size Darcy's law gives a pack, and the
    mean flow with fluctuations (float64, on the GPU)."""
    g = _gen(seed + 7919)
    ubar = 1e-3 if case["geometry"] == "duct" else 1e-4
    a = int((mask[0] == 0).sum())
    grad = 6e-5 if case["geometry"] == "duct" else 3e-5
    nz = case["nz"]
    z = torch.arange(nz, device="cuda", dtype=torch.float64)
    pore = (mask == 0).double()
    noise = torch.randn((4,) + tuple(mask.shape), generator=g, device="cuda", dtype=torch.float32).double()
    rho = 1 + (grad * (nz - 1 - z))[:, None, None] + 0.02 * grad * noise[0]
    u = torch.stack([0.3 * ubar * noise[1], 0.3 * ubar * noise[2], ubar * (2 + 0.3 * noise[3])]) * pore
    return ubar * a, rho, u


def _members(case, seed):
    # the edges are the case's own, spread over its range, both ends among them; the packs come from the seed
    r = np.random.RandomState(1000 * case["members"] + case["lo"] + case["hi"])
    sizes = [[int(v) for v in np.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"] + 1), 3))]
             for _ in range(case["members"])]
    sizes[0] = [case["lo"]] * 3
    sizes[-1] = [case["hi"], case["hi"] - 1, case["hi"]]
    masks = [_pack(s[0], s[1], max(12, s[2]), 31 * seed + k, reservoir=3) for k, s in enumerate(sizes)]
    return masks, [1e-4 * int((m[0] == 0).sum()) for m in masks]


def _colour_start(case, seed):
    """mask, phase field (the injected fluid in the inlet reservoir with a rough front) and flux."""
    mask = _pack(case["nx"], case["ny"], case["nz"], seed, rmin=5.0, rmax=10.0)
    g = _gen(seed + 104729)
    front = 4 + 4 * torch.rand(case["ny"], case["nx"], generator=g, device="cuda", dtype=torch.float64)
    z = torch.arange(case["nz"], device="cuda", dtype=torch.float64)[:, None, None]
    return mask, torch.tanh(front[None] - z), 2e-4 * int((mask[0] == 0).sum())


ALPHA, BETA, PHI_S = 0.01, 0.95, -1.0


def _conv_tensors(case, seed):
    """Padded BF16 activation rows (ReLU outputs, zero border), the second operand and He-scaled weights."""
    g = _gen(seed)
    b, x, y, z, ci, co, op = (case[k] for k in ("batch", "nx", "ny", "nz", "cin", "cout", "op"))

    def rows(c, relu):
        t = torch.zeros(b, z + 2, y + 2, x + 2, c, device="cuda", dtype=torch.bfloat16)
        v = torch.randn(b, z, y, x, c, generator=g, device="cuda")
        t[:, 1:-1, 1:-1, 1:-1] = (v.relu() if relu else 0.1 * v).bfloat16()
        return t

    inp = rows(co, False) if op == 1 else rows(ci, True)
    aux = rows(co, False) if op == 2 else None
    w = (torch.randn(co, 27, ci, generator=g, device="cuda") * math.sqrt(2 / (27 * ci))).bfloat16()
    bias = 0.1 * torch.randn(co, generator=g, device="cuda")
    return inp, aux, w, bias


def _net_params(net_shapes, n, seed):
    r = np.random.RandomState((seed + 13) % (1 << 31))
    p = np.zeros(n, np.float32)
    k = 0
    for co, ci in net_shapes:
        m = co * ci * 27
        p[k:k + m] = r.standard_normal(m).astype(np.float32) * math.sqrt(2 / (27 * ci))
        p[k + m:k + m + co] = 0.05 * r.standard_normal(co)
        k += m + co
    return p


def _net_shapes(levels, base):
    c = [base << l for l in range(levels)]
    s = [(c[0], 1), (c[0], c[0])]
    for l in range(1, levels):
        s += [(c[l], c[l - 1]), (c[l], c[l])]
    for l in range(levels - 2, -1, -1):
        s += [(c[l], c[l + 1]), (c[l], c[l])]
    return s + [(4, c[0])]


def _grad_inputs(case, seed):
    """Interior crops of packs and their targets: u / u_D and the scaled pressure drop of a plane (NaN: no target)."""
    b, x, y, z = (case[k] for k in ("batch", "nx", "ny", "nz"))
    masks = torch.stack([_pack(x, y, z, 17 * seed + k, porosity=0.38, rmin=8.0, rmax=16.0, reservoir=0) for k in range(b)])
    g = _gen(seed + 3)
    t = torch.randn(b, 4, z, y, x, generator=g, device="cuda") * 0.8
    t[:, 2] += 1.5
    t[:, 3] = 1.4 + 0.5 * torch.randn(b, z, 1, 1, generator=g, device="cuda")
    pore = masks == 0
    t *= pore[:, None]
    t[:, 3][~pore] = float("nan")
    t[:, 3, -1] = float("nan")
    return masks.cpu().numpy(), t.cpu().numpy()


# ------------------------------------------------------------------- cases ---
def prepare(case, seed):
    kind = case["kind"]
    stream = torch.cuda.current_stream()
    s = {"case": case}
    if kind == "flow":
        mask = _flow_mask(case, seed)
        q, rho, u = _flow_start(case, mask, seed)
        lat = Lattice(mask.cpu().numpy(), case["tau"], "mrt", case["precision"], stream=stream)
        lat.set_kernel(case["variant"])
        lat.set_flux_bc(q)
        lat.set_fields(rho.cpu().numpy(), *u.cpu().numpy())
        s["lat"] = lat
        if case["precision"] != "fp64":
            s["rho"] = torch.empty(tuple(mask.shape), device="cuda", dtype=torch.float32)
            s["u"] = torch.empty((3,) + tuple(mask.shape), device="cuda", dtype=torch.float32)
    elif kind == "ensemble":
        masks, qs = _members(case, seed)
        b = Batch([m.cpu().numpy() for m in masks], case["tau"], "mrt", case["precision"], stream=stream)
        b.set_config(1)  # per-step launches at the 48-register cap: what the library's autotuner picks
        for k, q in enumerate(qs):
            b.set_flux_bc(k, q)
        s["batch"] = b
    elif kind == "colour":
        mask, phi, q = _colour_start(case, seed)
        c = ColorLattice(mask.cpu().numpy(), case["tau"], ALPHA, BETA, PHI_S, case["precision"], stream=stream)
        c.set_phase(phi.cpu().numpy())
        c.set_flux_bc(q, 1.0)
        s["colour"] = c
    elif kind == "conv":
        inp, aux, w, bias = _conv_tensors(case, seed)
        shape = tuple(inp.shape[:4])
        out = (torch.empty(shape + (case["cout"],), device="cuda", dtype=torch.bfloat16) if case["op"] == 0 else
               torch.empty(shape + (case["cin"],), device="cuda", dtype=torch.bfloat16) if case["op"] == 1 else
               torch.empty_like(w, dtype=torch.float32))
        s.update(inp=inp, aux=aux, w=w, bias=bias, out=out, stream=stream)
    else:
        net = WarmStartNet(case["levels"], case["base"], stream=stream)
        net.set_params(_net_params(net.layer_shapes(), net.n_params, seed))
        s["net"] = net
        if kind == "grad":
            s["masks"], s["targets"] = _grad_inputs(case, seed)
        else:
            s["mask"] = _pack(case["nx"], case["ny"], case["nz"], seed, rmin=8.0, rmax=16.0).cpu().numpy()
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "flow":
        lat = s["lat"]
        lat.step(case["steps"])
        out = {}
        if case["sample"]:  # the convergence loop's check: outlet flux and inlet density
            out["q_out"] = lat.get_flux(5)[0]
            out["rho_in"] = lat.get_flux(4)[1]
        if case["precision"] == "fp64":
            out["rho"], ux, uy, uz = lat.fields()
            out["u"] = [ux, uy, uz]
        else:
            lat.fields_device(s["rho"], s["u"])
            out["rho"], out["u"] = s["rho"], s["u"]
        return out
    if kind == "ensemble":
        b = s["batch"]
        b.step(case["steps"])
        # kept as float32, as the training data of the warm start are
        out = []
        for k in range(len(b)):
            rho, ux, uy, uz = b.fields(k)
            out.append({"rho": rho.astype(np.float32), "u": np.stack([ux, uy, uz]).astype(np.float32)})
        return out
    if kind == "colour":
        s["colour"].step(case["steps"])
        kept = np.float64 if case["precision"] == "fp64" else np.float32
        rho, ux, uy, uz, phi = s["colour"].fields()
        return {"rho": rho.astype(kept), "u": np.stack([ux, uy, uz]).astype(kept), "phi": phi.astype(kept)}
    if kind == "conv":
        if case["op"] == 2:
            s["out"].zero_()  # a weight gradient is added to the buffer
        conv3d_bf16(case["op"], s["inp"].data_ptr(), s["aux"].data_ptr() if case["op"] == 2 else 0, s["w"].data_ptr(),
                    s["bias"].data_ptr() if case["op"] == 0 else 0, case["op"] == 0, s["out"].data_ptr(), case["batch"],
                    case["nx"], case["ny"], case["nz"], case["cin"], case["cout"], stream=s["stream"])
        return s["out"]
    if kind == "grad":
        loss, g = s["net"].loss_grad(s["masks"], s["targets"])
        return {"loss": loss, "grad": g}
    return s["net"].predict(s["mask"])


def work(case):
    kind = case["kind"]
    if kind == "ensemble":
        mid = (case["lo"] + case["hi"]) / 2
        cells = case["members"] * mid ** 3
        n = 0.38 * cells
        return {"bytes": case["steps"] * n * 38 * BYTES[case["precision"]] + 16 * cells, "flops": case["steps"] * n * 200}
    cells = case["nx"] * case["ny"] * case["nz"]
    if kind == "flow":
        n = (case["nx"] - 2) * (case["ny"] - 2) * case["nz"] if case["geometry"] == "duct" else 0.38 * cells
        out = 32 if case["precision"] == "fp64" else 16
        return {"bytes": case["steps"] * n * 38 * BYTES[case["precision"]] + out * cells, "flops": case["steps"] * n * 200}
    if kind == "colour":  # momentum 19 in and out, two phases 7 in and out each
        n = 0.38 * cells
        return {"bytes": case["steps"] * n * 66 * BYTES[case["precision"]] + 20 * cells, "flops": case["steps"] * n * 400}
    if kind == "conv":
        v = case["batch"] * cells
        io = v * 2 * (case["cin"] + case["cout"])
        return {"bytes": io + (2 if case["op"] < 2 else 4) * 27 * case["cin"] * case["cout"],
                "flops": 2 * 27 * case["cin"] * case["cout"] * v}
    shapes = _net_shapes(case["levels"], case["base"])
    level = [0, 0] + [l for l in range(1, case["levels"]) for _ in (0, 1)]
    level += [l for l in range(case["levels"] - 2, -1, -1) for _ in (0, 1)] + [0]
    fwd = sum(2 * 27 * co * ci * cells / 8 ** l for (co, ci), l in zip(shapes, level))
    params = sum(co * ci * 27 + co for co, ci in shapes)
    if kind == "grad":
        return {"bytes": case["batch"] * cells * 17 + 4 * params + 2 * params, "flops": 3 * case["batch"] * fwd}
    return {"bytes": cells * 17 + 2 * params, "flops": fwd}


# ------------------------------------------------ the same in 64 bits (torch) ---
class _Nodes:
    """Pore list of a mask and, per direction, the node that a value streaming in direction q comes from."""

    def __init__(self, mask):
        nz, ny, nx = mask.shape
        self.shape = (nz, ny, nx)
        grid = torch.full((nz + 2, ny + 2, nx + 2), -3, dtype=torch.int64, device="cuda")  # -3: beyond a z face
        grid[1:-1] = -2                                                                    # -2: beyond a lateral face
        grid[1:-1, 1:-1, 1:-1] = -1                                                        # -1: solid
        self.pore = mask == 0
        self.n = int(self.pore.sum())
        inner = grid[1:-1, 1:-1, 1:-1]
        inner[self.pore] = torch.arange(self.n, device="cuda")
        flat = grid.reshape(-1)
        at = torch.nonzero(torch.nn.functional.pad(self.pore, (1, 1, 1, 1, 1, 1)).reshape(-1))[:, 0]
        sy, sz = nx + 2, (nx + 2) * (ny + 2)
        self.src = [flat[at - (c[2] * sz + c[1] * sy + c[0])] for c in XI]
        self.a_in = int(self.pore[0].sum())
        self.a_out = int(self.pore[-1].sum())

    def stream_index(self, nq):
        """Flat index into (nq, n) of the value that arrives in each direction (halfway bounce-back at walls)."""
        own = torch.arange(self.n, device="cuda")
        opp = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, nq)]
        return torch.stack([torch.where(self.src[q] >= 0, q * self.n + self.src[q], opp[q] * self.n + own)
                            for q in range(nq)])

    def dense(self, v):
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        out[self.pore] = v
        return out


def _moments(d):
    rho = d.sum(0)
    j = [sum(XI[q][a] * d[q] for q in range(19) if XI[q][a]) for a in range(3)]
    return rho, j


def _close(d, sl, rho, inlet, q_flux):
    """Pressure (or flux) closure of Appendix B on the nodes `sl`, shifted distributions; returns rho - 1 used."""
    e = d[:, sl]
    flat = e[0] + e[1] + e[2] + e[3] + e[4] + e[7] + e[8] + e[9] + e[10]
    nx = 0.5 * (e[1] + e[7] + e[9] - e[2] - e[10] - e[8])
    ny = 0.5 * (e[3] + e[7] + e[10] - e[4] - e[9] - e[8])
    if inlet:
        known = flat + 2 * (e[6] + e[12] + e[13] + e[16] + e[17])
        if q_flux is not None:
            rho = (q_flux + known.sum()) / known.numel()
        uz = rho - known
        e[5], e[11], e[14] = e[6] + uz / 3, e[12] + uz / 6 - nx, e[13] + uz / 6 + nx
        e[15], e[18] = e[16] + uz / 6 - ny, e[17] + uz / 6 + ny
    else:
        uz = flat + 2 * (e[5] + e[11] + e[14] + e[15] + e[18]) - rho
        e[6], e[12], e[13] = e[5] - uz / 3, e[11] - uz / 6 + nx, e[14] - uz / 6 - nx
        e[16], e[17] = e[15] - uz / 6 + ny, e[18] - uz / 6 - ny
    return rho


def _relax(d, sp, sm, add=None):
    rho, (ux, uy, uz) = _moments(d)
    uu = 1.5 * (ux * ux + uy * uy + uz * uz)
    out = torch.empty_like(d)
    out[0] = d[0] - sp * (d[0] - W[0] * (rho - uu))
    for q in range(1, 19, 2):
        xu = sum(c * v for c, v in zip(XI[q], (ux, uy, uz)) if c)
        p = sp * (0.5 * (d[q] + d[q + 1]) - W[q] * (rho + 4.5 * xu * xu - uu))
        m = sm * (0.5 * (d[q] - d[q + 1]) - W[q] * 3 * xu)
        out[q] = d[q] - p - m
        out[q + 1] = d[q + 1] - p + m
    return out


def _flow64(mask, tau, q_flux, steps, rho=None, u=None):
    """Lattice.step from f_eq(rho, u) (rest if None): density and velocity after `steps`, dense, and the samples."""
    nd = _Nodes(mask)
    sp = 1 / tau
    sm = 8 * (2 - sp) / (8 - sp)
    d = torch.zeros(19, nd.n, dtype=torch.float64, device="cuda")
    if rho is not None:
        r = rho[nd.pore] - 1
        v = [c[nd.pore] for c in u]
        uu = 1.5 * sum(c * c for c in v)
        for q in range(19):
            xu = sum(c * w for c, w in zip(XI[q], v))
            d[q] = W[q] * (r + 3 * xu + 4.5 * xu * xu - uu)
    idx = nd.stream_index(19)
    rho_in = 0.0
    for _ in range(steps):
        d = d.reshape(-1)[idx]
        rho_in = _close(d, slice(0, nd.a_in), None, True, q_flux)
        _close(d, slice(nd.n - nd.a_out, nd.n), 0.0, False, None)
        d = _relax(d, sp, sm)
    dr, j = _moments(d)
    return nd.dense(1 + dr), [nd.dense(c) for c in j], float(j[2][nd.n - nd.a_out:].sum()), 1 + float(rho_in)


def _colour64(mask, phi, q_flux, tau, steps):
    nd = _Nodes(mask)
    n = nd.n
    sp = 1 / tau
    sm = 8 * (2 - sp) / (8 - sp)
    w7 = [1 / 3] + [1 / 9] * 6
    ph = phi[nd.pore]
    d = torch.zeros(19, n, dtype=torch.float64, device="cuda")
    a = torch.stack([w * (1 + ph) / 2 for w in w7])
    b = torch.stack([w * (1 - ph) / 2 for w in w7])
    idx, idx7 = nd.stream_index(19), nd.stream_index(7)
    own = torch.arange(n, device="cuda")
    # neighbour x + xi_q is the source of the opposite direction
    nbr = [None] + [nd.src[q + 1 if q % 2 else q - 1] for q in range(1, 19)]
    safe = [None] + [torch.where(v >= 0, v, own) for v in nbr[1:]]
    solid = [None] + [v == -1 for v in nbr[1:]]
    inl, outl = slice(0, nd.a_in), slice(n - nd.a_out, n)
    for _ in range(steps):
        a[5, inl] = 0
        b[5, inl] = 0
        a[5, inl] = 1.0 - a[:, inl].sum(0)
        b[5, inl] = 0.0 - b[:, inl].sum(0)
        na, nb = a.sum(0), b.sum(0)
        ph = (na - nb) / (na + nb)
        c = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(3)]
        for q in range(1, 19):
            v = torch.where(solid[q], PHI_S, ph[safe[q]])
            for k in range(3):
                if XI[q][k]:
                    c[k] += 3 * W[q] * XI[q][k] * v
        mag = torch.sqrt(c[0] ** 2 + c[1] ** 2 + c[2] ** 2)
        inv = torch.where(mag > 0, 1 / torch.where(mag > 0, mag, 1.0), 0.0)
        nv = [x * inv for x in c]
        d = d.reshape(-1)[idx]
        _close(d, inl, None, True, q_flux)
        _close(d, outl, 0.0, False, None)
        _, j = _moments(d)
        am = ALPHA * mag
        dm = {1: am, 9: 0.5 * am * (2 * nv[0] ** 2 - nv[1] ** 2 - nv[2] ** 2), 11: 0.5 * am * (nv[1] ** 2 - nv[2] ** 2),
              13: 0.5 * am * nv[0] * nv[1], 14: 0.5 * am * nv[1] * nv[2], 15: 0.5 * am * nv[0] * nv[2]}
        d = _relax(d, sp, sm)
        for k, m in dm.items():
            row = [19 * sum(x * x for x in e) - 30 if k == 1 else 3 * e[0] ** 2 - sum(x * x for x in e) if k == 9 else
                   e[1] ** 2 - e[2] ** 2 if k == 11 else e[0] * e[1] if k == 13 else e[1] * e[2] if k == 14 else e[0] * e[2]
                   for e in XI]
            norm = sum(r * r for r in row)
            for q in range(19):
                if row[q]:
                    d[q] += (sp * row[q] / norm) * m
        oa, ob = torch.empty_like(a), torch.empty_like(b)
        for q in range(7):
            xu = sum(e * v for e, v in zip(XI[q], j) if e)
            xn = sum(e * v for e, v in zip(XI[q], nv) if e)
            oa[q] = w7[q] * na * (1 + 4.5 * xu + BETA * nb * xn)
            ob[q] = w7[q] * nb * (1 + 4.5 * xu - BETA * na * xn)
        a, b = oa.reshape(-1)[idx7], ob.reshape(-1)[idx7]
        a[5, inl] = 0
        b[5, inl] = 0
        a[6, outl] = w7[6] * na[outl] * (1 - 4.5 * j[2][outl])
        b[6, outl] = w7[6] * nb[outl] * (1 - 4.5 * j[2][outl])
    dr, j = _moments(d)
    na, nb = a.sum(0), b.sum(0)
    return {"rho": nd.dense(1 + dr), "u": torch.stack([nd.dense(v) for v in j]), "phi": nd.dense((na - nb) / (na + nb))}


def _shifted(x, t):
    """Rows of the padded layout at tap t, zero outside."""
    dz, dy, dx = t // 9 - 1, (t // 3) % 3 - 1, t % 3 - 1
    off = (dz * x.shape[2] + dy) * x.shape[3] + dx
    flat = x.reshape(-1, x.shape[4])
    out = torch.zeros_like(flat)
    if off >= 0:
        out[:flat.shape[0] - off] = flat[off:]
    else:
        out[-off:] = flat[:off]
    return out


def _conv64(case, seed):
    inp, aux, w, bias = _conv_tensors(case, seed)
    x, w = inp.double(), w.double()
    inner = torch.zeros(x.shape[:4], dtype=torch.bool, device="cuda")
    inner[:, 1:-1, 1:-1, 1:-1] = True
    if case["op"] == 2:
        g = aux.double().reshape(-1, case["cout"])
        return torch.stack([g.t() @ _shifted(x, t) for t in range(27)], 1)
    fwd = case["op"] == 0
    out = sum(_shifted(x, t if fwd else 26 - t) @ (w[:, t].t() if fwd else w[:, t]) for t in range(27))
    if fwd:
        out = (out + bias.double()).relu()
    return (out * inner.reshape(-1, 1)).reshape(x.shape[:4] + (out.shape[1],))


def _net64(params, masks, levels, base):
    """The network's outputs [B][4][z][y][x] from float64 parameters and uint8 masks (differentiable)."""
    import torch.nn.functional as F
    layers, k = [], 0
    for co, ci in _net_shapes(levels, base):
        m = co * ci * 27
        w = params[k:k + m].reshape(co, 27, ci).permute(0, 2, 1).reshape(co, ci, 3, 3, 3)
        layers.append((w, params[k + m:k + m + co]))
        k += m + co
    it = iter(layers)

    def conv(v):
        w, b = next(it)
        return F.conv3d(v, w, b, padding=1)

    x = (masks == 0).double()[:, None]
    e = [conv(conv(x).relu()).relu()]
    for _ in range(1, levels):
        e.append(conv(conv(F.avg_pool3d(e[-1], 2)).relu()).relu())
    v = e[-1]
    for l in range(levels - 2, -1, -1):
        v = conv(conv(F.interpolate(v, scale_factor=2, mode="nearest")).relu() + e[l]).relu()
    return conv(v) * x


def exact(case, seed):
    kind = case["kind"]
    if kind == "flow":
        mask = _flow_mask(case, seed)
        q, rho, u = _flow_start(case, mask, seed)
        r, v, q_out, rho_in = _flow64(mask, case["tau"], q, case["steps"], rho, u)
        out = {"q_out": q_out, "rho_in": rho_in} if case["sample"] else {}
        out["rho"] = r
        out["u"] = v if case["precision"] == "fp64" else torch.stack(v)
        return out
    if kind == "ensemble":
        masks, qs = _members(case, seed)
        if case["steps"] * sum(float((m == 0).sum()) for m in masks) > 6e9:
            return None
        got = [_flow64(m, case["tau"], q, case["steps"]) for m, q in zip(masks, qs)]
        return [{"rho": r, "u": torch.stack(v)} for r, v, _, _ in got]
    if kind == "colour":
        mask, phi, q = _colour_start(case, seed)
        return _colour64(mask, phi, q, case["tau"], case["steps"])
    if kind == "conv":
        return _conv64(case, seed)
    shapes = _net_shapes(case["levels"], case["base"])
    n = sum(co * ci * 27 + co for co, ci in shapes)
    p = torch.from_numpy(_net_params(shapes, n, seed)).cuda().double()
    if kind == "grad":
        m, t = _grad_inputs(case, seed)
        masks, t = torch.from_numpy(m).cuda(), torch.from_numpy(t).cuda().double()
        pores = int((masks == 0).sum())
        p.requires_grad_(True)
        total = 0.0
        for k in range(case["batch"]):  # one sample at a time: the sum over samples is the batch's loss
            d = _net64(p, masks[k:k + 1], case["levels"], case["base"]) - torch.nan_to_num(t[k:k + 1])
            d = d * ~torch.isnan(t[k:k + 1]) * (masks[k:k + 1] == 0)[:, None]
            loss = d.square().sum() / (4 * pores)
            loss.backward()
            total += float(loss)
        return {"loss": total, "grad": p.grad}
    mask = _pack(case["nx"], case["ny"], case["nz"], seed, rmin=8.0, rmax=16.0)
    with torch.no_grad():
        return _net64(p, mask[None], case["levels"], case["base"])[0]
