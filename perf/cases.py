"""Work that a user of this package has it do, as cases that can be timed and compared.

A case names one call (its "kind") with its grid and options:

  evaluate   Magnet.set_target once, then Magnet.evaluate(rho) -> J, dJ/drho: one objective and
             gradient for an optimiser of the user's own
  step       Magnet.evaluate_step: one iteration of the projected-gradient loop (optimize.Run)
  field      Magnet.stray_field(rho) -> H on the whole grid
  autograd   StrayField.apply and its backward for a dense cotangent dL/dH
  oneshot    Magnet.objective_and_gradient(rho, mask, Ht): nothing prepared, H returned too
  lbfgsb     lbfgsb.optimize_magnet: the first iterations of the paper's minimiser
  batch      batch.BatchedRuns.run(10): ten steps of several specifications side by side
  conv_fwd   tmn_conv3d_forward: one convolution layer of the warm-start network
  conv_bwd   tmn_conv3d_backward_weight and _data: the gradients of such a layer

Grids: (nx, ny, nz) output cells, the design is the slab z < nzd, the target a tw x th patch on
the top `planes` planes. J is returned as float32: it is a sum over a float32 field.
"""

import ctypes
import math

import numpy as np
import torch

from paper_1707_09898_gb300 import Magnet, StrayField, _lib
from paper_1707_09898_gb300 import workloads as W
from paper_1707_09898_gb300.batch import BatchedRuns
from paper_1707_09898_gb300.lbfgsb import optimize_magnet

DEV = torch.device("cuda", 0)
MS = 1.0 / (4e-7 * math.pi)  # 1 T / mu0, A/m
ALPHA = 0.1                  # the step of the projected-gradient loop
TILTED = (0.48, -0.6, 0.64)
BATCH_STEPS = 10


def grid(kind, name, n, nzd, planes=1, tw=None, th=None, m0="z", w="z", ht="const", p=3.0, **more):
    return dict({"name": name, "kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "nzd": nzd, "planes": planes,
                 "tw": tw or max(1, n[0] // 4), "th": th or max(1, n[1] // 4), "m0": m0, "w": w, "ht": ht, "p": p}, **more)


def conv(kind, name, batch, dhw, cin, cout):
    return {"name": name, "kind": kind, "batch": batch, "d": dhw[0], "h": dhw[1], "w": dhw[2], "cin": cin, "cout": cout}


def listed():
    return [
        # the smallest grid that is documented (16^3 design, one layer of target cells): an outer
        # optimiser that wants J and the gradient on the host calls this; launches and latency count
        grid("evaluate", "evaluate 16x16x17", (16, 16, 17), 16, tw=4, th=4),
        # the paper's validation problem (39^3 cube, two target planes, 62,361 cells) with its
        # minimiser: eight iterations of L-BFGS-B from a start of the user's own
        grid("lbfgsb", "L-BFGS-B 39x39x41", (39, 39, 41), 39, planes=2, tw=5, th=5, w="minus_half_z", iters=8),
        # a 64^3 design optimised by optimize.Run, which reads J after every step
        grid("step", "step 64x64x72", (64, 64, 72), 64, tw=16, th=16, sync=True),
        # sixteen 64^3 specifications optimised side by side
        {"name": "batch 16 of 64x64x72", "kind": "batch", "specs": 16},
        # throughput of the loop at 128^3 and 256^3: steps queued one after another, J not waited for
        grid("step", "step 128x128x128", (128, 128, 128), 128, sync=False),
        grid("step", "step 256x256x256", (256, 256, 256), 256, sync=False),
        # a magnetization that varies from cell to cell and a target for all three components
        grid("evaluate", "evaluate 128x128x66 varying M0", (128, 128, 66), 64, tw=32, th=32, m0="vmf", w="xyz", ht="field"),
        # the field of a finished design on the whole grid
        grid("field", "field 256x256x256", (256, 256, 256), 256),
        # a user's own loss on the field, differentiated by autograd, on an odd grid
        grid("autograd", "autograd 150x101x77", (150, 101, 77), 60, m0="tilted"),
        # one call with nothing prepared, H wanted for inspection, a target with a full field
        grid("oneshot", "one-shot 192x160x100", (192, 160, 100), 90, planes=4, m0="tilted", w="xyz", ht="field"),
        # the widest full-resolution layer of the warm-start network, inference and training
        conv("conv_fwd", "conv forward 48-16", 2, (64, 64, 64), 48, 16),
        conv("conv_bwd", "conv backward 48-16", 2, (64, 64, 64), 48, 16),
    ]


def log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


LAYERS = ((16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (96, 32), (48, 16))


def draw(rng):
    kind = rng.choice(("evaluate", "evaluate", "step", "step", "field", "autograd", "oneshot", "lbfgsb", "batch", "conv_fwd",
                       "conv_bwd"))
    if kind.startswith("conv"):
        cin, cout = rng.choice(LAYERS)
        # rows as the network has them (a power of two) or as another grid would
        side = rng.choice((8, 16, 32, 64)) if rng.random() < 0.7 else rng.randint(8, 60)
        c = conv(kind, "", rng.randint(1, 4), (log_int(rng, 8, 64), log_int(rng, 8, 64), side), cin, cout)
    elif kind == "batch":
        c = {"kind": kind, "specs": rng.randint(4, 16)}
    elif kind == "lbfgsb":
        n = rng.randint(24, 48)
        c = grid(kind, "", (n, rng.randint(24, 48), n + 2), n, planes=rng.randint(1, 2), tw=rng.randint(4, 9),
                 th=rng.randint(4, 9), w="minus_half_z", iters=rng.randint(4, 8))
    else:
        m0 = rng.choice(("z", "z", "tilted", "vmf"))
        w = rng.choice(("z", "z", "xyz"))
        most = 2 ** 21 if m0 == "vmf" or w == "xyz" else 2 ** 24
        cells = math.exp(rng.uniform(math.log(16 ** 3), math.log(most)))
        while True:  # a box of about so many cells, no axis more than four times another
            r = [math.exp(rng.uniform(-0.69, 0.69)) for _ in range(3)]
            s = (cells / (r[0] * r[1] * r[2])) ** (1.0 / 3.0)
            n = [int(round(s * v)) for v in r]
            if all(8 <= v <= 256 for v in n) and n[0] * n[1] * n[2] <= most:
                break
        nzd = rng.randint(max(1, (3 * n[2]) // 4), n[2])
        c = grid(kind, "", n, nzd, planes=min(n[2], rng.choice((1, 1, 2, 5, 12))), tw=rng.randint(1, n[0]),
                 th=rng.randint(1, n[1]), m0=m0, w=w, ht=rng.choice(("const", "field")),
                 p=rng.choice((3.0, 3.0, 2.0, 1.0)))
        if kind == "step":
            c["sync"] = rng.random() < 0.5
    c.pop("name", None)
    return c


# -- inputs ---------------------------------------------------------------------------
def generator(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def density(shape, g):
    """Densities as a loop meets them: the box constraint is active in a third of the cells."""
    return (torch.rand(shape, generator=g, device=DEV) * 1.5 - 0.25).clamp_(0.0, 1.0)


def inputs(c, seed):
    """Plain tensors and numbers of a grid case, from the seed alone."""
    g = generator(seed)
    nx, ny, nz, nzd = c["nx"], c["ny"], c["nz"], c["nzd"]
    out = {"rho": density((nzd, ny, nx), g), "M0": tuple(MS * v for v in ((0.0, 0.0, 1.0) if c["m0"] == "z" else TILTED)),
           "w": {"z": (0.0, 0.0, 1.0), "xyz": (1.0, 0.5, 2.0), "minus_half_z": (0.0, 0.0, -0.5)}[c["w"]],
           "Htc": (0.0, 0.0, 0.2 * MS), "Ht": None}
    if c["kind"] == "lbfgsb":
        # the paper's units, M0 = 1; densities off the bounds so that every breakpoint is passed
        out.update(M0=(0.0, 0.0, 1.0), Htc=(0.0, 0.0, 0.0), rho=0.6 + 0.3 * torch.rand((nzd, ny, nx), generator=g, device=DEV))
    if c["m0"] == "vmf":  # scattered about +z
        v = torch.randn((3, nzd, ny, nx), generator=g, device=DEV) * 0.3
        v[2] += 1.0
        out["M0"] = (MS * v / v.norm(dim=0)).contiguous()
    mask = torch.zeros((nz, ny, nx), dtype=torch.uint8, device=DEV)
    x0, y0 = (nx - c["tw"]) // 2, (ny - c["th"]) // 2
    mask[nz - c["planes"]:, y0:y0 + c["th"], x0:x0 + c["tw"]] = 1
    out["mask"] = mask
    if c["ht"] == "field":
        out["Ht"] = (torch.randn((3, nz, ny, nx), generator=g, device=DEV) * (0.05 * MS) * mask).contiguous()
    if c["kind"] == "autograd":
        out["gH"] = torch.randn((3, nz, ny, nx), generator=g, device=DEV)
    return out


def conv_inputs(c, seed):
    g = generator(seed)
    dims = (c["batch"], c["d"], c["h"], c["w"])
    cin, cout = c["cin"], c["cout"]
    x = torch.randn(dims + (cin,), generator=g, device=DEV).relu_().to(torch.bfloat16)  # activations follow a ReLU
    wt = torch.randn((27, cin, cout), generator=g, device=DEV) * math.sqrt(2.0 / (27 * cin))
    b = torch.randn((cout,), generator=g, device=DEV) * 0.1
    gout = torch.randn(dims + (cout,), generator=g, device=DEV) * 1e-3 if c["kind"] == "conv_bwd" else None
    if gout is not None:
        gout *= torch.rand(gout.shape, generator=g, device=DEV) < 0.5  # masked by the layer's ReLU
    return dims, x, wt, b, gout


def specs(c, seed):
    return [W.config5(100000 + 1000 * (int(seed) % 1000) + i) for i in range(c["specs"])]


# -- what a program holds before the call ------------------------------------------------
def prepare(case, seed):
    c = case
    if c["kind"].startswith("conv"):
        dims, x, wt, b, gout = conv_inputs(c, seed)
        L = _lib.lib()
        s = {"case": c, "L": L, "dims": dims, "x": x, "w": wt, "b": b, "gout": gout}
        for k in ("wf", "wb"):
            s[k] = torch.empty((27 * c["cin"] * c["cout"],), dtype=torch.bfloat16, device=DEV)
        ok(L.tmn_pack_conv_weights(ptr(wt), ptr(s["wf"]), ptr(s["wb"]), c["cin"], c["cout"], stream()))
        if c["kind"] == "conv_fwd":
            s["out"] = torch.empty(dims + (c["cout"],), dtype=torch.bfloat16, device=DEV)
        else:  # the scratch that WarmStartNet allocates for a layer's weight gradient
            n = L.tmn_conv3d_backward_weight_work(math.prod(dims), c["cin"], c["cout"]) + 8 * 160 * 128 * 64
            s["work"] = torch.empty((n,), dtype=torch.float32, device=DEV)
            s["dw"], s["db"] = torch.empty_like(wt), torch.empty_like(b)
            s["din"] = torch.empty(dims + (c["cin"],), dtype=torch.float32, device=DEV)
        return s
    if c["kind"] == "batch":
        return {"case": c, "runs": BatchedRuns(specs(c, seed), device=0, steps_per_graph=BATCH_STEPS)}
    s = inputs(c, seed)
    s["case"] = c
    m = Magnet((c["nx"], c["ny"], c["nz"]), c["nzd"], M0=s["M0"], p=c["p"], device=0)
    s["m"] = m
    if c["kind"] in ("evaluate", "step", "lbfgsb"):
        m.set_target(s["mask"], Ht=s["Ht"], Ht_const=s["Htc"], w=s["w"])
        s["G"] = torch.empty_like(s["rho"])
    if c["kind"] == "step":  # a loop starts with one evaluation, which gives the first gradient
        m.evaluate(s["rho"], G=s["G"])
    if c["kind"] == "oneshot":
        s["G"] = torch.empty_like(s["rho"])
        s["H"] = torch.empty((3, c["nz"], c["ny"], c["nx"]), device=DEV)
    if c["kind"] == "field":
        s["H"] = torch.empty((3, c["nz"], c["ny"], c["nx"]), device=DEV)
    if c["kind"] == "autograd":
        s["rho"].requires_grad_(True)
    return s


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream(DEV).cuda_stream)


def ok(code):
    if code != 0:
        raise RuntimeError("the call returned %d" % code)


# -- one pass ------------------------------------------------------------------------------
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "evaluate":
        J, G = s["m"].evaluate(s["rho"], G=s["G"])
        return {"J": np.float32(J), "G": G}
    if kind == "step":
        J, G = s["m"].evaluate_step(s["rho"], s["G"], ALPHA, sync=c["sync"])
        out = {"rho": s["rho"], "G": G}
        if c["sync"]:
            out["J"] = np.float32(J)
        return out
    if kind == "field":
        return {"H": s["m"].stray_field(s["rho"], out=s["H"])}
    if kind == "autograd":
        H = StrayField.apply(s["rho"], s["m"])
        return {"H": H, "grad": torch.autograd.grad(H, s["rho"], s["gH"])[0]}
    if kind == "oneshot":
        J, G = s["m"].objective_and_gradient(s["rho"], s["mask"], Ht=s["Ht"], Ht_const=s["Htc"], w=s["w"], G=s["G"],
                                             H_out=s["H"])
        return {"J": np.float32(J), "G": G, "H": s["H"]}
    if kind == "lbfgsb":
        r = optimize_magnet(s["m"], s["rho"], maxiter=c["iters"])
        return {"x": r.x, "f": np.asarray(r.history, np.float32)}
    if kind == "batch":
        s["runs"].run(BATCH_STEPS)
        return {"rho": list(s["runs"].rho)}
    L, dims, cin, cout = s["L"], s["dims"], c["cin"], c["cout"]
    if kind == "conv_fwd":
        ok(L.tmn_conv3d_forward(ptr(s["x"]), ptr(s["wf"]), ptr(s["b"]), ptr(s["out"]), *dims, cin, cout, 1, stream()))
        return {"out": s["out"]}
    ok(L.tmn_conv3d_backward_weight(ptr(s["x"]), ptr(s["gout"]), ptr(s["dw"]), ptr(s["db"]), ptr(s["work"]),
                                    s["work"].numel(), *dims, cin, cout, stream()))
    ok(L.tmn_conv3d_backward_data(ptr(s["gout"]), ptr(s["wb"]), ptr(s["din"]), *dims, cin, cout, 0, stream()))
    return {"dw": s["dw"], "db": s["db"], "din": s["din"]}


# -- what a pass cannot do without -------------------------------------------------------------
def fft_flops(c, spectra):
    """Real transforms of the doubled box, 2.5 N log2 N each."""
    n = 8.0 * c["nx"] * c["ny"] * c["nz"]
    return 2.5 * n * math.log2(n) * spectra


def work(case):
    """Inputs read once, outputs written once, the convolution by FFT (or the layer's products)."""
    c = case
    if c["kind"].startswith("conv"):
        vox = float(c["batch"] * c["d"] * c["h"] * c["w"])
        macs = vox * 27 * c["cin"] * c["cout"]
        wts = 27.0 * c["cin"] * c["cout"]
        if c["kind"] == "conv_fwd":
            return {"bytes": 2 * vox * (c["cin"] + c["cout"]) + 2 * wts, "flops": 2 * macs}
        return {"bytes": vox * (2 * c["cin"] + 4 * c["cout"] + 4 * c["cin"]) + 6 * wts, "flops": 4 * macs}
    if c["kind"] == "batch":
        g = {"nx": 64, "ny": 64, "nz": 72}
        return {"bytes": c["specs"] * BATCH_STEPS * 64.0 ** 3 * 12, "flops": c["specs"] * BATCH_STEPS * fft_flops(g, 4)}
    out = float(c["nx"] * c["ny"] * c["nz"])
    design = float(c["nx"] * c["ny"] * c["nzd"])
    m0 = 12.0 * design if c["m0"] == "vmf" else 0.0
    nin = 3 if c["m0"] == "vmf" else 1
    nw = 3 if c["w"] == "xyz" else 1
    target = c["planes"] * c["tw"] * c["th"] * (1.0 + (4.0 * nw if c["ht"] == "field" else 0.0))
    if c["kind"] == "field":
        return {"bytes": 4 * design + m0 + 12 * out, "flops": fft_flops(c, nin + 3)}
    if c["kind"] == "autograd":
        return {"bytes": 8 * design + m0 + 24 * out, "flops": fft_flops(c, 2 * (nin + 3))}
    if c["kind"] == "oneshot":
        return {"bytes": 8 * design + m0 + 12 * out + out + target, "flops": fft_flops(c, nin + 3 + nw + nin)}
    one = {"bytes": (16.0 if c["kind"] == "step" else 8.0) * design + m0 + target, "flops": fft_flops(c, 2 * nin + 2 * nw)}
    if c["kind"] == "lbfgsb":  # an evaluation and a few vector passes an iteration
        return {k: (c["iters"] + 1) * v for k, v in one.items()}
    return one


# -- the same in 64 bits ---------------------------------------------------------------------------
F64 = torch.float64


def newell_f(x, y, z):
    """Newell, Williams and Dunlop (1993): the function whose second differences give N_xx."""
    x, y, z = x.abs(), y.abs(), z.abs()
    x2, y2, z2 = x * x, y * y, z * z
    r = (x2 + y2 + z2).sqrt()
    tiny = torch.finfo(F64).tiny
    a = torch.where(y > 0, 0.5 * y * (z2 - x2) * torch.asinh(y / (x2 + z2).sqrt().clamp_min(tiny)), 0.0)
    b = torch.where(z > 0, 0.5 * z * (y2 - x2) * torch.asinh(z / (x2 + y2).sqrt().clamp_min(tiny)), 0.0)
    a = torch.where((x2 + z2) > 0, a, 0.0)
    b = torch.where((x2 + y2) > 0, b, 0.0)
    t = torch.where((x > 0) & (y > 0) & (z > 0), x * y * z * torch.atan(y * z / (x * r).clamp_min(tiny)), 0.0)
    return (2 * x2 - y2 - z2) * r / 6 + a + b - t


def newell_g(x, y, z):
    """The same for N_xy: odd in x and y, even in z."""
    sign = torch.sign(x) * torch.sign(y)
    x, y, z = x.abs(), y.abs(), z.abs()
    x2, y2, z2 = x * x, y * y, z * z
    r = (x2 + y2 + z2).sqrt()
    xs, ys, zs = x.clamp_min(1e-300), y.clamp_min(1e-300), z.clamp_min(1e-300)
    v = -x * y * r / 3
    v = v + x * y * z * torch.asinh(z / (xs * xs + ys * ys).sqrt())
    v = v + y / 6 * (3 * z2 - y2) * torch.asinh(x / (ys * ys + z2).sqrt())
    v = v + x / 6 * (3 * z2 - x2) * torch.asinh(y / (xs * xs + z2).sqrt())
    t = z2 * z / 6 * torch.atan(x * y / (zs * r)) + z * y2 / 2 * torch.atan(x * z / (ys * r)) + z * x2 / 2 * torch.atan(y * z / (xs * r))
    v = v - torch.where(z > 0, t, 0.0)
    return torch.where((x > 0) & (y > 0), sign * v, 0.0)


def newell(i, j, k):
    """The six tensor components (xx, yy, zz, xy, xz, yz) of cubic unit cells at integer offsets."""
    out = [0.0] * 6
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            for e in (-1, 0, 1):
                wt = (2.0 if a == 0 else -1.0) * (2.0 if b == 0 else -1.0) * (2.0 if e == 0 else -1.0) / (4 * math.pi)
                x, y, z = i + a, j + b, k + e
                for n, v in enumerate((newell_f(x, y, z), newell_f(y, x, z), newell_f(z, y, x), newell_g(x, y, z),
                                       newell_g(x, z, y), newell_g(y, z, x))):
                    out[n] = out[n] + wt * v
    return torch.stack(out)


def far(i, j, k, comp):
    """One component of the dipole kernel averaged over both cells: the rule with nodes 0 and
    +-sqrt(2/5) and weights 7/12 and 5/24 on an axis is exact to the fifth moment, and the closed
    form above loses its digits at this distance."""
    node, rows = math.sqrt(0.4), ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))
    p, q = rows[comp]
    out = 0.0
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            for e in (-1, 0, 1):
                wt = math.prod(7 / 12 if v == 0 else 5 / 24 for v in (a, b, e)) / (4 * math.pi)
                r = (i + a * node, j + b * node, k + e * node)
                r2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
                inv = 1.0 / r2.sqrt()
                i3 = inv * inv * inv
                out = out + wt * ((i3 if p == q else 0.0) - 3 * i3 * inv * inv * r[p] * r[q])
    return out


class Operator:
    """H = -N * M by the zero-padded transform in 64 bits (cubic cells)."""

    NEAR = 16
    ODD = ((0, 0, 0), (0, 0, 0), (0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))  # (x, y, z) of each component
    AT = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}

    def __init__(self, nx, ny, nz):
        self.n = (nz, ny, nx)
        self.L = tuple(next(v for v in range(2 * n, 4 * n + 2) if smooth(v)) for n in self.n)
        k, j, i = torch.meshgrid(*(torch.arange(min(n, self.NEAR + 1), device=DEV, dtype=F64) for n in self.n), indexing="ij")
        self.near = newell(i, j, k)
        self.kept = {}

    def spectrum(self, comp):
        if comp in self.kept:
            return self.kept[comp]
        k, j, i = (torch.arange(n, device=DEV, dtype=F64) for n in self.n)
        octant = torch.empty(self.n, device=DEV, dtype=F64)
        for a in range(0, self.n[0], 16):  # some planes at a time
            octant[a:a + 16] = far(i[None, None], j[None, :, None], k[a:a + 16, None, None], comp)
        nn = self.near[comp]
        octant[:nn.shape[0], :nn.shape[1], :nn.shape[2]] = nn
        full = octant
        for axis in range(3):  # the other octants by symmetry, zeros between
            sign = -1.0 if self.ODD[comp][2 - axis] else 1.0
            mirrored = sign * full.flip(axis).narrow(axis, 0, self.n[axis] - 1)
            shape = list(full.shape)
            shape[axis] = self.L[axis] - 2 * self.n[axis] + 1
            full = torch.cat((full, torch.zeros(shape, device=DEV, dtype=F64), mirrored), axis)
        s = torch.fft.rfftn(full)
        if s.numel() <= 1 << 24:  # the large ones are made again
            self.kept[comp] = s
        return s

    def __call__(self, src, nout, wanted=(0, 1, 2)):
        """-(N * src) on the lowest nout planes; src: three arrays, or None for zero."""
        given = [(b, torch.fft.rfftn(v.to(F64), s=self.L)) for b, v in enumerate(src) if v is not None]
        out = []
        for a in range(3):
            if a not in wanted:
                out.append(None)
                continue
            acc = 0.0
            for b, f in given:
                acc = acc + self.spectrum(self.AT[(min(a, b), max(a, b))]) * f
            out.append(-torch.fft.irfftn(acc, s=self.L)[:nout, :self.n[1], :self.n[2]])
            del acc
        return out


def smooth(v):
    if v % 2:
        return False
    for f in (2, 3, 5, 7):
        while v % f == 0:
            v //= f
    return v == 1


def components(M0):
    return [M0[a].to(F64) if isinstance(M0, torch.Tensor) else (M0[a] if M0[a] != 0.0 else None) for a in range(3)]


def field(op, rho, M0, p, nz, wanted=(0, 1, 2)):
    q = rho.to(F64) ** p
    return op([None if m is None else m * q for m in components(M0)], nz, wanted)


def chain(op, rho, M0, p, gH, nzd):
    """p rho^(p-1) M0 . D(gH)"""
    m = components(M0)
    back = op(gH, nzd, [a for a in range(3) if m[a] is not None])
    return p * rho.to(F64) ** (p - 1) * sum(m[a] * back[a] for a in range(3) if m[a] is not None)


def objective(op, rho, M0, p, mask, Ht, Htc, w):
    """J, dJ/drho of sum_mask sum_c w_c (H_c - Ht_c)^2."""
    wanted = [a for a in range(3) if w[a] != 0.0]
    H = field(op, rho, M0, p, mask.shape[0], wanted)
    J, g = 0.0, [None] * 3
    for a in wanted:
        t = Ht[a].to(F64) if Ht is not None else float(np.float32(Htc[a]))
        d = (H[a] - t) * mask
        J = J + w[a] * (d * d).sum()
        g[a] = 2 * w[a] * d
    return J, chain(op, rho, M0, p, g, rho.shape[0])


def stepped(rho, G):
    return (rho - ALPHA * G / G.abs().max()).clamp(0.0, 1.0)


def convolve(x, wt):
    """3x3x3, zero padding 1: x [N][D][H][W][Cin], wt [27][Cin][Cout] in 64 bits."""
    n, d, h, w, _ = x.shape
    xp = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    out = 0.0
    for t in range(27):
        dz, dy, dx = t // 9, t // 3 % 3, t % 3
        out = out + xp[:, dz:dz + d, dy:dy + h, dx:dx + w] @ wt[t]
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "lbfgsb":  # several line searches: there is no closed value
        return None
    if c["kind"].startswith("conv"):
        dims, x, wt, b, gout = conv_inputs(c, seed)
        w64 = wt.to(torch.bfloat16).to(F64)  # a layer's products take its bfloat16 copies
        if c["kind"] == "conv_fwd":
            return {"out": (convolve(x.to(F64), w64) + b.to(F64)).relu()}
        g64 = gout.to(torch.bfloat16).to(F64)
        d, h, w = dims[1:]
        xp = torch.nn.functional.pad(x.to(F64), (0, 0, 1, 1, 1, 1, 1, 1))
        flat = g64.reshape(-1, c["cout"])
        dw = torch.stack([xp[:, t // 9:t // 9 + d, t // 3 % 3:t // 3 % 3 + h, t % 3:t % 3 + w].reshape(-1, c["cin"]).T @ flat
                          for t in range(27)])
        return {"dw": dw, "db": gout.to(F64).reshape(-1, c["cout"]).sum(0), "din": convolve(g64, w64.flip(0).transpose(1, 2))}
    if c["kind"] == "batch":
        out, op = [], Operator(64, 64, 72)
        for wl in specs(c, seed):
            rho = torch.full((64, 64, 64), 0.5, device=DEV, dtype=F64)
            mask = torch.from_numpy(wl.mask()).to(DEV)
            htc = [float(v) for v in wl.Ht_const_vec()]
            for _ in range(BATCH_STEPS):
                rho = stepped(rho, objective(op, rho, tuple(float(v) for v in wl.M0_const()), wl.p, mask, None, htc, wl.w)[1])
            out.append(rho)
        return {"rho": out}
    s = inputs(c, seed)
    op = Operator(c["nx"], c["ny"], c["nz"])
    args = (op, s["rho"], s["M0"], c["p"])
    if c["kind"] == "field":
        return {"H": torch.stack(field(*args, c["nz"]))}
    if c["kind"] == "autograd":
        return {"H": torch.stack(field(*args, c["nz"])), "grad": chain(*args, list(s["gH"]), c["nzd"])}
    goal = (s["mask"], s["Ht"], s["Htc"], s["w"])
    J, G = objective(*args, *goal)
    if c["kind"] == "evaluate":
        return {"J": J, "G": G}
    if c["kind"] == "oneshot":
        return {"J": J, "G": G, "H": torch.stack(field(*args, c["nz"]))}
    rho = stepped(s["rho"].to(F64), G)
    J, G = objective(op, rho, s["M0"], c["p"], *goal)
    return {"rho": rho, "G": G, **({"J": J} if c["sync"] else {})}
