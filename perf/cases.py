"""What the speed of this library is judged by: calls that its users make, over the sizes they make them at.

Four families, each through the public Python entry points:
  lattice  one D2Q9 lattice: fields in (smrt_init_macros), n updates (smrt_step), fields out
           (smrt_macros) and, where a run watches for its steady state, smrt_residual;
  batch    many cavities of uneven size advanced together (smrt_batch_step on a tuned batch), or a
           whole data set of small cavities made from nothing (create, autotune, run, read back);
  unet     the warm-start network: one recorded training step, or one prediction;
  conv     one of its 3x3 layers: forward with bias and SiLU, input gradient, weight gradient.
"""
import math

import numpy as np
import torch

import paper_2409_01076_gb300 as S
from paper_2409_01076_gb300 import nn as K
from paper_2409_01076_gb300 import unet as U
from paper_2409_01076_gb300 import workloads as W

DEV = "cuda"
U_LID = 0.1
BC = {"cavity": W.CAVITY, "periodic": W.ALL_PERIODIC, "couette": W.COUETTE, "channel": W.CHANNEL}
PREC = {"f64": S.SMRT_PREC_F64, "f32": S.SMRT_PREC_F32, "f16": S.SMRT_PREC_F16, "bf16": S.SMRT_PREC_BF16}
LAYOUT = {"ab": S.SMRT_LAYOUT_AB, "aa": S.SMRT_LAYOUT_AA}
COLLISION = {"smrt": S.SMRT_COLLISION_SMRT, "srt": S.SMRT_COLLISION_SRT, "two_tau": S.SMRT_COLLISION_TWO_TAU}
ELEM = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
TAU_S = 0.9                                     # the free second relaxation time of the two-tau form
FLOPS = 90                                      # of one node update


def lattice(name, nx, ny, flow, re, steps, prec="f32", layout="ab", collision="smrt", rounding="nearest",
            residual=False):
    return {"name": name, "family": "lattice", "nx": nx, "ny": ny, "flow": flow, "re": re, "steps": steps,
            "prec": prec, "layout": layout, "collision": collision, "rounding": rounding, "residual": residual}


def listed():
    return [
        # the validation cavity, far from filling the chip: 2,000 updates that wait for one another
        lattice("cavity_64_f64", 64, 64, "cavity", 100.0, 2000, "f64"),
        # one leg of a run to the steady state in 64 bits at the learned warm start's size, with its check
        lattice("steady_256_f64", 256, 256, "cavity", 1000.0, 500, "f64", residual=True),
        # the same at the size the warm start is transferred to, in 32 bits: 1,000 updates, then the check
        lattice("steady_1024_f32", 1024, 1024, "cavity", 1000.0, 1000, residual=True),
        # a ragged channel between a resting floor and a moving top, by the comparison collision
        lattice("couette_1021x509_f32_srt", 1021, 509, "couette", 500.0, 300, collision="srt"),
        # the headline throughput run
        lattice("tgv_8192_f32", 8192, 8192, "periodic", 100000.0, 20),
        # a large cavity in the one-buffer layout
        lattice("cavity_4096_f32_aa", 4096, 4096, "cavity", 10000.0, 100, layout="aa"),
        # a large cavity in 16-bit storage
        lattice("cavity_8192_f16", 8192, 8192, "cavity", 5000.0, 40, "f16"),
        # hundreds of cavities of uneven size and Reynolds number on their way to the steady state
        {"name": "batch_mix_512", "family": "batch", "count": 512, "lo": 64, "hi": 1024, "steps": 50},
        # a small training set, from the list of Reynolds numbers to the fields
        {"name": "dataset_192x128", "family": "dataset", "count": 192, "n": 128, "steps": 400},
        # one training step of the warm-start network at its training size and batch
        {"name": "unet_train_16x256", "family": "unet_train", "batch": 16, "n": 256},
        # the prediction in front of one warm start
        {"name": "unet_predict_1x256", "family": "unet_predict", "batch": 1, "n": 256},
        # one of its middle layers, forward and backward
        {"name": "conv_16x128x128_64", "family": "conv", "batch": 16, "h": 128, "w": 128, "cin": 64, "cout": 64},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["lattice"] * 6 + ["batch", "dataset", "unet_train", "unet_predict", "conv", "conv"])
    if kind == "lattice":
        prec = rng.choice(["f64", "f32", "f32", "f32", "f16", "bf16"])
        top = 1024 if prec == "f64" else 8192
        nx, ny = size(32, top), size(32, top)
        if rng.random() < 0.4:
            ny = nx
        flow = rng.choice(sorted(BC))
        most = (1e8 if prec == "f64" else 1.5e9) / (nx * ny)
        steps = max(2, min(2000, int(most), size(10, 2000)))
        side = min(nx, ny)                      # a Reynolds number that this side resolves
        re = min(max(math.exp(rng.uniform(math.log(100.0), math.log(5000.0))), side / 4.0), 4.0 * side)
        return dict(lattice("", nx, ny, flow, round(re, 1), steps, prec,
                            rng.choice(["ab", "ab", "aa"]), rng.choice(["smrt", "smrt", "srt", "two_tau"]),
                            rng.choice(["nearest", "stochastic"]) if prec in ("f16", "bf16") else "nearest",
                            prec in ("f64", "f32") and rng.random() < 0.5), name="drawn")
    if kind == "batch":
        lo = rng.choice([32, 48, 64, 100])
        return {"name": "drawn", "family": "batch", "count": size(16, 512), "lo": lo, "hi": size(4 * lo, 1024),
                "steps": size(10, 50)}
    if kind == "dataset":
        n = size(48, 256)
        return {"name": "drawn", "family": "dataset", "count": size(16, max(17, 192 * 128 * 128 // (n * n))), "n": n,
                "steps": 100 * rng.randint(1, 4)}
    if kind == "unet_train":
        return {"name": "drawn", "family": "unet_train", "batch": rng.randint(1, 16), "n": 8 * rng.randint(8, 32)}
    if kind == "unet_predict":
        return {"name": "drawn", "family": "unet_predict", "batch": rng.randint(1, 8), "n": 8 * rng.randint(8, 32)}
    cin, cout = (rng.choice([16, 32, 64, 96, 128, 192, 256, 384]), rng.choice([32, 64, 128, 256]))
    h, w = size(16, 256), size(16, 256)
    most = 16 * 256 * 256 * 64 * 64 // (h * w * cin * cout)
    return {"name": "drawn", "family": "conv", "batch": max(1, min(rng.randint(1, 16), most)), "h": h, "w": w,
            "cin": cin, "cout": cout}


# ---- inputs --------------------------------------------------------------------------------------

def generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def initial_fields(nx, ny, flow, seed):
    """A smooth flow: a few random vortex modes (at rest on every wall), |u| up to about 0.06, rho within 1 %."""
    g = generator(seed)
    x = (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) / nx
    y = (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) / ny
    wall_x, wall_y = flow == "cavity", flow != "periodic"
    u = torch.zeros(2, ny, nx, dtype=torch.float64, device=DEV)
    rho = torch.ones(ny, nx, dtype=torch.float64, device=DEV)
    for k in range(3):
        r = torch.rand(6, generator=g, device=DEV, dtype=torch.float64).tolist()
        amp, px, py = 0.02 * (0.5 + r[0]), 2 * math.pi * r[1], 2 * math.pi * r[2]
        mx, my = 1 + int(3 * r[3]), 1 + int(3 * r[4])
        ax = 2 * math.pi * mx * x + px
        ay = 2 * math.pi * my * y + py
        ex = torch.sin(math.pi * x) ** 2 if wall_x else torch.ones_like(x)
        ey = torch.sin(math.pi * y) ** 2 if wall_y else torch.ones_like(y)
        u[0] -= amp * torch.outer(ey * torch.sin(ay), ex * torch.cos(ax))
        u[1] += amp * torch.outer(ey * torch.cos(ay), ex * torch.sin(ax))
        rho += 0.003 * (r[5] - 0.5) * torch.outer(torch.cos(ay), torch.cos(ax))
    return rho, u


def u_lid_of(case):
    return U_LID if case["flow"] in ("cavity", "couette") else 0.0


def tau_of(case):
    return W.cavity_tau(min(case["nx"], case["ny"]), U_LID, case["re"])


def batch_of(case, seed):
    """(sides, relaxation times) of a batch: the sides by the case, the Reynolds numbers by the seed."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    if case["family"] == "dataset":
        re = np.exp(rng.uniform(math.log(100.0), math.log(min(10000.0, 40.0 * case["n"])), size=case["count"]))
        sides = [case["n"]] * case["count"]
    else:
        sides = []
        while not sides or sides[-1] * 2 <= case["hi"]:
            sides.append(sides[-1] * 2 if sides else case["lo"])
        sides = [n for n, _ in W.batched_cavities(case["count"], case["count"], sides)]
        re = np.exp(rng.uniform(math.log(100.0), math.log(5000.0), size=case["count"]))
    return sides, [W.cavity_tau(n, U_LID, float(r)) for n, r in zip(sides, re)]


def unet_weights(seed):
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    p = {}
    for name, ci, co, k, _ in U.LAYERS:
        ci = 3 if ci == "in" else 32 * ci
        co = 3 if co == "out" else 32 * co
        p[name + ".w"] = rng.normal(0.0, math.sqrt(2.0 / (ci * k * k)), size=(co, k * k * ci)).astype(np.float32)
        p[name + ".b"] = rng.normal(0.0, 0.05, size=(co,)).astype(np.float32)
    return p


def unet_inputs(case, seed):
    """Network input (N, n, n, 3) and a smooth target of the size the steady fields have."""
    rng = np.random.Generator(np.random.PCG64(int(seed) + 1))
    res = np.exp(rng.uniform(math.log(U.RE_LO), math.log(U.RE_HI), size=case["batch"])).tolist()
    x = U.input_grid(res, case["n"], case["n"])
    gx, gy, re = x[..., 1], x[..., 2], x[..., 0]
    t = torch.stack([torch.sin(math.pi * gx) * (gy ** (2 + 4 * re) - 0.3 * gy),
                     0.5 * torch.sin(2 * math.pi * gx) * torch.sin(math.pi * gy) * (1 - 0.4 * re),
                     0.2 * (gx - 0.5) * gy], dim=-1).contiguous()
    return x, t


def conv_inputs(case, seed):
    """Activations, weights, bias and output gradient; what tensor cores read is already a half value."""
    g = generator(seed)
    n, h, w, ci, co = (case[k] for k in ("batch", "h", "w", "cin", "cout"))

    def normal(*shape, scale=1.0):
        return scale * torch.randn(*shape, generator=g, device=DEV)

    x = torch.nn.functional.silu(normal(n, h, w, ci)).half().float()
    wt = normal(co, 9 * ci, scale=math.sqrt(2.0 / (9 * ci))).half().float()
    dz = normal(n, h, w, co, scale=0.1).half().float()
    return x, wt, normal(co, scale=0.05), dz


# ---- preparing and running -----------------------------------------------------------------------

def prepare(case, seed):
    return {"lattice": prepare_lattice, "batch": prepare_batch, "dataset": prepare_dataset,
            "unet_train": prepare_unet, "unet_predict": prepare_unet, "conv": prepare_conv}[case["family"]](case, seed)


def run(state):
    return state["run"](state)


def prepare_lattice(case, seed):
    nx, ny = case["nx"], case["ny"]
    h = S.smrt_create(nx, ny, tau_of(case), u_lid_of(case), BC[case["flow"]])
    S.smrt_set_option(h, S.SMRT_OPT_PRECISION, PREC[case["prec"]])
    S.smrt_set_option(h, S.SMRT_OPT_LAYOUT, LAYOUT[case["layout"]])
    S.smrt_set_option(h, S.SMRT_OPT_COLLISION, COLLISION[case["collision"]])
    S.smrt_set_option(h, S.SMRT_OPT_TAU_S, TAU_S)
    if case["rounding"] == "stochastic":
        S.smrt_set_option(h, S.SMRT_OPT_ROUNDING, S.SMRT_ROUND_STOCHASTIC)
    rho, u = initial_fields(nx, ny, case["flow"], seed)
    return {"run": run_lattice, "h": h, "steps": case["steps"], "residual": case["residual"], "rho": rho, "u": u,
            "rho_out": torch.empty_like(rho), "u_out": torch.empty_like(u)}


def run_lattice(s):
    S.smrt_init_macros(s["h"], s["rho"], s["u"])
    S.smrt_step(s["h"], s["steps"])
    out = {}
    if s["residual"]:
        r, sums = S.smrt_residual(s["h"])
        out = {"residual": r, "mass": sums[0]}
    S.smrt_macros(s["h"], s["rho_out"], s["u_out"])
    return dict(out, rho=s["rho_out"], u=s["u_out"])


def field_views(sides):
    """One buffer for every lattice's (rho, u), and its views."""
    flat = torch.empty(sum(3 * n * n for n in sides), dtype=torch.float64, device=DEV)
    views, at = [], 0
    for n in sides:
        views.append((flat[at:at + n * n].view(n, n), flat[at + n * n:at + 3 * n * n].view(2, n, n)))
        at += 3 * n * n
    return flat, views


def prepare_batch(case, seed):
    sides, taus = batch_of(case, seed)
    b = S.smrt_batch_create(sides, sides, taus, [U_LID] * len(sides))
    S.smrt_batch_autotune(b, 6)
    flat, views = field_views(sides)
    return {"run": run_batch, "b": b, "steps": case["steps"], "flat": flat, "views": views}


def run_batch(s):
    """The cavities go on from where the last pass left them, as a user's do."""
    S.smrt_batch_step(s["b"], s["steps"])
    for k, (rho, u) in enumerate(s["views"]):
        S.smrt_batch_macros(s["b"], k, rho, u)
    return s["flat"]


def prepare_dataset(case, seed):
    sides, taus = batch_of(case, seed)
    flat, views = field_views(sides)
    return {"run": run_dataset, "sides": sides, "taus": taus, "steps": case["steps"], "flat": flat, "views": views}


def run_dataset(s):
    b = S.smrt_batch_create(s["sides"], s["sides"], s["taus"], [U_LID] * len(s["sides"]))
    S.smrt_batch_autotune(b, 6)
    S.smrt_batch_run(b, 1e-7, 100, s["steps"], S.SMRT_BATCH_RESIDUAL_STRIDE)
    steps, res, _ = S.smrt_batch_status(b)
    for k, (rho, u) in enumerate(s["views"]):
        S.smrt_batch_macros(b, k, rho, u)
    S.smrt_batch_destroy(b)
    return {"fields": s["flat"], "residual": res, "steps": steps}


def prepare_unet(case, seed):
    net = U.UNet(base=32)
    net.load_numpy(unet_weights(seed))
    x, t = unet_inputs(case, seed)
    if case["family"] == "unet_predict":
        return {"run": lambda s: s["net"].predict(s["x"]), "net": net, "x": x}
    net.capture(x, t)
    return {"run": run_train, "net": net}


def run_train(s):
    y = s["net"].replay()
    return {"y": y, "grads": s["net"].grads}


def prepare_conv(case, seed):
    x, wt, bias, dz = conv_inputs(case, seed)
    n, h, w, ci, co = (case[k] for k in ("batch", "h", "w", "cin", "cout"))
    half = dict(dtype=torch.float16, device=DEV)
    xb, dzb = torch.empty(x.numel(), **half), torch.empty(dz.numel(), **half)
    K.smrt_nn_to_half_blocked(x, xb)
    K.smrt_nn_to_half_blocked(dz, dzb)
    wp, wpa = (torch.empty(K.smrt_nn_pack3_halves(*s), **half) for s in ((co, ci), (ci, co)))
    K.smrt_nn_pack3_many([(wt, wp, K.SMRT_NN_PACK_FORWARD, co, ci, ci), (wt, wpa, K.SMRT_NN_PACK_ADJOINT, co, ci, ci)])
    return {"run": run_conv, "xb": xb, "dzb": dzb, "wp": wp, "wpa": wpa, "bias": bias, "in": (n, h, w, ci),
            "out": (n, h, w, co), "z": torch.empty(n, h, w, co, device=DEV),
            "ab": torch.empty(n * h * w * co, **half), "dx": torch.empty(n, h, w, ci, device=DEV),
            "gw": torch.empty(co, 9 * ci, device=DEV), "err": torch.zeros(1, dtype=torch.int32, device=DEV)}


def run_conv(s):
    ci, co = s["in"][3], s["out"][3]
    K.smrt_nn_conv3_tma_bias_act(s["xb"], s["in"], s["wp"], co, s["bias"], 1, s["z"], None, s["ab"], s["err"])
    K.smrt_nn_conv3_tma(s["dzb"], s["out"], s["wpa"], s["dx"], ci, 1.0, 0.0, s["err"])
    s["gw"].zero_()
    K.smrt_nn_conv3_wgrad_tma(s["xb"], s["in"], s["dzb"], co, s["gw"], 1.0, s["err"])
    return {"z": s["z"], "ab": s["ab"], "dx": s["dx"], "gw": s["gw"]}


# ---- work ----------------------------------------------------------------------------------------

def conv_flops(case):
    return 2.0 * case["batch"] * case["h"] * case["w"] * 9 * case["cin"] * case["cout"]


def unet_flops(batch, n):
    total, side = 0.0, {"enc1": n, "enc2": n // 2, "enc3": n // 4, "mida": n // 8, "midb": n // 8,
                        "dec3": n // 4, "dec2": n // 2, "dec1": n, "head": n}
    for name, ci, co, k, _ in U.LAYERS:
        ci = 3 if ci == "in" else 32 * ci
        co = 3 if co == "out" else 32 * co
        total += 2.0 * batch * side[name[:4]] ** 2 * k * k * ci * co
    return total


def work(case):
    f = case["family"]
    if f == "lattice":      # fields in, the state once, fields out
        n = case["nx"] * case["ny"]
        return {"bytes": n * (48 + 9 * ELEM[case["prec"]]), "flops": FLOPS * n * case["steps"]}
    if f in ("batch", "dataset"):
        n = sum(s * s for s in batch_of(case, 0)[0])
        return {"bytes": n * (24 + (72 if f == "batch" else 36)), "flops": FLOPS * n * case["steps"]}
    if f == "conv":
        px = case["batch"] * case["h"] * case["w"]
        return {"bytes": px * (2 * case["cin"] + 2 * case["cout"] + 6 * case["cout"] + 4 * case["cin"])
                + case["cin"] * case["cout"] * 9 * 8, "flops": 3 * conv_flops(case)}
    px, params = case["batch"] * case["n"] ** 2, 4 * 1.95e6
    if f == "unet_predict":
        return {"bytes": px * 24 + params, "flops": unet_flops(case["batch"], case["n"])}
    return {"bytes": px * 36 + 2 * params, "flops": 3 * unet_flops(case["batch"], case["n"])}


# ---- the same in 64 bits, by torch alone -----------------------------------------------------------

EX, EY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class Exact:
    """The update of the listed flows on f[9][ny][nx] (or a stack [9][count][ny][nx]), straight from the paper."""

    def __init__(self, flow, tau, u_lid, collision):
        self.flow, self.tau, self.u_lid, self.collision = flow, tau, u_lid, collision

    @staticmethod
    def equilibrium(rho, ux, uy):
        uu = 1.5 * (ux * ux + uy * uy)
        out = []
        for a in range(9):
            eu = EX[a] * ux + EY[a] * uy
            out.append(WT[a] * rho * (1 + 3 * eu + 4.5 * eu * eu - uu))
        return torch.stack(out)

    @staticmethod
    def macros(f):
        rho = f.sum(0)
        ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
        uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
        return rho, ux, uy

    def step(self, f):
        q = self.equilibrium(*self.macros(f))
        n = f - q
        p1, p2 = n[1] - n[2] + n[3] - n[4], n[5] - n[6] + n[7] - n[8]
        inv = 1 / self.tau
        if self.collision == "srt":
            post = f - n * inv
        else:
            ts = 1.0 if self.collision == "smrt" else 1 / TAU_S
            post = f - n * ts
            for a in range(1, 9):
                post[a] += (1 if a % 2 else -1) * (ts - inv) / 4 * (p1 if a < 5 else p2)
        out = torch.empty_like(f)
        for a in range(9):
            out[a] = torch.roll(post[a], (EY[a], EX[a]), (-2, -1))
            if self.flow == "cavity" and EX[a]:
                i = 0 if EX[a] > 0 else -1
                out[a][..., :, i] = post[OPP[a]][..., :, i]
            if self.flow != "periodic" and EY[a]:
                j = 0 if EY[a] > 0 else -1
                lid = self.u_lid if EY[a] < 0 and self.flow in ("cavity", "couette") else 0.0
                out[a][..., j, :] = post[OPP[a]][..., j, :] + 6 * WT[a] * EX[a] * lid
        return out


def exact(case, seed):
    return {"lattice": exact_lattice, "batch": exact_batch, "dataset": exact_dataset, "unet_train": exact_unet,
            "unet_predict": exact_unet, "conv": exact_conv}[case["family"]](case, seed)


def exact_lattice(case, seed):
    rho, u = initial_fields(case["nx"], case["ny"], case["flow"], seed)
    e = Exact(case["flow"], tau_of(case), u_lid_of(case), case["collision"])
    f = e.equilibrium(rho, u[0], u[1])
    for _ in range(case["steps"]):
        f = e.step(f)
    rho, ux, uy = e.macros(f)
    out = {"rho": rho, "u": torch.stack([ux, uy])}
    if case["residual"]:
        _, vx, vy = e.macros(e.step(f))
        r = ((vx - ux).square().sum() + (vy - uy).square().sum()).sqrt() / (vx.square().sum() + vy.square().sum()).sqrt()
        out = dict(out, residual=float(r), mass=float(rho.sum()))
    return out


def exact_cavities(sides, taus, steps, stride):
    """(rho, u) of every cavity after `steps` updates from rest, and its change over the last `stride`."""
    fields, change = [None] * len(sides), [0.0] * len(sides)
    for n in sorted(set(sides)):
        same = [k for k, m in enumerate(sides) if m == n]
        most = max(1, int(2e7) // (n * n))
        for at in range(0, len(same), most):
            ks = same[at:at + most]
            tau = torch.tensor([taus[k] for k in ks], dtype=torch.float64, device=DEV).view(-1, 1, 1)
            e = Exact("cavity", tau, U_LID, "smrt")
            one = torch.ones(len(ks), n, n, dtype=torch.float64, device=DEV)
            f = e.equilibrium(one, 0 * one, 0 * one)
            for t in range(steps):
                if t == steps - stride:
                    _, px, py = e.macros(f)
                f = e.step(f)
            rho, ux, uy = e.macros(f)
            num = ((ux - px).square() + (uy - py).square()).sum((1, 2)).sqrt()
            den = (ux.square() + uy.square()).sum((1, 2)).sqrt()
            for j, k in enumerate(ks):
                fields[k] = torch.cat([rho[j].reshape(-1), ux[j].reshape(-1), uy[j].reshape(-1)])
                change[k] = float(num[j] / den[j]) / stride
    return torch.cat(fields), np.array(change)


def exact_batch(case, seed):
    sides, taus = batch_of(case, seed)
    return exact_cavities(sides, taus, case["steps"], 1)[0]


def exact_dataset(case, seed):
    sides, taus = batch_of(case, seed)
    fields, change = exact_cavities(sides, taus, case["steps"], 100)
    return {"fields": fields, "residual": change if case["steps"] > 100 else None, "steps": None}


def nchw(w, k):
    co = w.shape[0]
    return w.view(co, k, k, -1).permute(0, 3, 1, 2)


def exact_unet(case, seed):
    F = torch.nn.functional
    train = case["family"] == "unet_train"
    p = {k: torch.tensor(v, dtype=torch.float64, device=DEV).requires_grad_(train)
         for k, v in unet_weights(seed).items()}
    x, t = unet_inputs(case, seed)

    def c(name, v):
        v = F.conv2d(v, nchw(p[name + ".w"], 3), p[name + ".b"], padding=1)
        return F.silu(v)

    def up(a, b):
        return torch.cat([F.interpolate(a, scale_factor=2, mode="nearest"), b], 1)

    with torch.set_grad_enabled(train):
        e1 = c("enc1b", c("enc1a", x.double().permute(0, 3, 1, 2)))
        e2 = c("enc2b", c("enc2a", F.avg_pool2d(e1, 2)))
        e3 = c("enc3b", c("enc3a", F.avg_pool2d(e2, 2)))
        m = c("midb", c("mida", F.avg_pool2d(e3, 2)))
        d3 = c("dec3b", c("dec3a", up(m, e3)))
        d2 = c("dec2b", c("dec2a", up(d3, e2)))
        d1 = c("dec1b", c("dec1a", up(d2, e1)))
        y = F.conv2d(d1, nchw(p["head.w"], 1), p["head.b"]).permute(0, 2, 3, 1)
        if not train:
            return y.contiguous()
        (2.0 ** 16 * F.mse_loss(y, t.double())).backward()
    return {"y": y.detach().contiguous(), "grads": {k: v.grad for k, v in p.items()}}


def exact_conv(case, seed):
    F = torch.nn.functional
    x, wt, bias, dz = (v.double() for v in conv_inputs(case, seed))
    n, h, w, ci, co = (case[k] for k in ("batch", "h", "w", "cin", "cout"))
    xc, zc, wc = x.permute(0, 3, 1, 2).contiguous(), dz.permute(0, 3, 1, 2).contiguous(), nchw(wt, 3).contiguous()
    z = F.conv2d(xc, wc, bias, padding=1)
    ab = F.silu(z).view(n, co // 8, 8, h, w).permute(0, 1, 3, 4, 2).reshape(-1)
    dx = F.conv_transpose2d(zc, wc, padding=1)
    gw = torch.empty(co, 3, 3, ci, dtype=torch.float64, device=DEV)
    pad = F.pad(xc, (1, 1, 1, 1))
    flat = zc.transpose(0, 1).reshape(co, -1)
    for ky in range(3):
        for kx in range(3):
            gw[:, ky, kx] = flat @ pad[:, :, ky:ky + h, kx:kx + w].transpose(0, 1).reshape(ci, -1).T
    return {"z": z.permute(0, 2, 3, 1).contiguous(), "ab": ab, "dx": dx.permute(0, 2, 3, 1).contiguous(),
            "gw": gw.view(co, 9 * ci)}
