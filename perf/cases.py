"""The work that users of this framework have it do, as measurable cases.

Four families, each called through the public classes of ``paper_2501_03759_gb300``:

  field2d  a periodic 2D field stepped by ``lbch.Solver`` (FP32, BF16- or FP16-deviation
           storage), phi read back on the device, mass and free energy logged where said;
  field3d  a periodic 3D field stepped by ``lbch.Solver3``, the snapshot kept in FP32;
  sweep    many uneven 2D fields stepped together by ``lbch.Batch``;
  leap     judged learned-leap cycles of ``lbnop.Surrogate`` on a 2D field;
  train    one optimiser step of ``lbnop.Surrogate`` on a batch of field pairs.

Sizes, strengths and initial fields are those of the repository's benchmark and tests (the
64^2 droplet, the 256^2 logged spinodal run, the 8192^2 field, the 512-field sweep, the
100^3 droplet and the 256^3 cube, the 512^2 leap), and for ``draw`` the ranges around them.

``exact`` evaluates the same quantities in FP64 with plain torch operations.
"""
import math
import os

import numpy as np
import torch

from paper_2501_03759_gb300 import lbch, lbnop

STORAGE = {"f32": lbch.STORE_F32, "bf16": lbch.STORE_BF16_DEV, "f16": lbch.STORE_F16_DEV}
# A full set of relaxation rates, as a user who tunes the MRT operator gives it.
OTHER_RATES = [1.0, 0.8, 1.3, 1.0, 1.6, 1.0, 0.7, 1.1, 1.5]
WEIGHTS = os.path.join(os.path.dirname(lbch.__file__), "weights", "leap512_k500.npy")
M, SIGMA, DW, EPS = 0.1, 0.01, 5.0, 0.03  # the defaults of make_params
LEAP_SCALE, LEAP_STEPS, LEAP_WARMUP, LR = 0.01, 500, 500, 1e-4


def listed():
    return [
        # The 64^2 droplet run, read out every 100 of its 2000 steps: launch-bound stepping.
        {"name": "droplet_64_logged", "kind": "field2d", "nx": 64, "ny": 64, "storage": "f32", "steps": 100,
         "ic": "droplet", "alpha": 0.3, "log": True, "rates": "default"},
        # The smallest call: one step at a time on a small field, phi watched after each.
        {"name": "watched_192x160", "kind": "field2d", "nx": 192, "ny": 160, "storage": "f32", "steps": 1,
         "ic": "droplet", "alpha": 0.3, "log": False, "rates": "default"},
        # The 256^2 spinodal run in 16-bit storage between two of its log lines.
        {"name": "spinodal_256_bf16", "kind": "field2d", "nx": 256, "ny": 256, "storage": "bf16", "steps": 100,
         "ic": "spinodal", "alpha": 0.2, "log": False, "rates": "default"},
        # A field cut to a measured domain: odd sizes, rows that are no multiple of any vector.
        {"name": "ragged_1001x517", "kind": "field2d", "nx": 1001, "ny": 517, "storage": "f32", "steps": 50,
         "ic": "spinodal", "alpha": 0.3, "log": False, "rates": "default"},
        # A user who tunes the relaxation rates, on a mid-size field in FP16 storage.
        {"name": "tuned_rates_2048_f16", "kind": "field2d", "nx": 2048, "ny": 2048, "storage": "f16", "steps": 20,
         "ic": "spinodal", "alpha": 0.3, "log": False, "rates": "other"},
        # The large single field in its two storages, with the energy reading of a log line.
        {"name": "spinodal_8192_f32", "kind": "field2d", "nx": 8192, "ny": 8192, "storage": "f32", "steps": 20,
         "ic": "spinodal", "alpha": 0.3, "log": False, "rates": "default"},
        {"name": "spinodal_8192_bf16", "kind": "field2d", "nx": 8192, "ny": 8192, "storage": "bf16", "steps": 20,
         "ic": "spinodal", "alpha": 0.3, "log": False, "rates": "default"},
        # The parameter sweep of 512 uneven fields between two snapshots.
        {"name": "sweep_512_fields", "kind": "sweep", "count": 512, "edges": "64,128,256,512", "storage": "f32",
         "steps": 50, "spec": 0},
        # The 3D droplet (100^3) and a cube for 3D coarsening, between two stored snapshots.
        {"name": "droplet_100_cubed", "kind": "field3d", "nx": 100, "ny": 100, "nz": 100, "steps": 400,
         "ic": "droplet", "alpha": 0.3},
        {"name": "spinodal_256_cubed", "kind": "field3d", "nx": 256, "ny": 256, "nz": 256, "steps": 400,
         "ic": "spinodal", "alpha": 0.3},
        # Surrogate-accelerated coarsening: judged, quarter-turn averaged leaps and correction steps.
        {"name": "leap_512", "kind": "leap", "n": 512, "turns": 4, "cycles": 2, "corr": 50, "alpha": 0.3},
        # One fine-tuning step of the leap network, as its training loop takes them.
        {"name": "train_512_b16", "kind": "train", "n": 512, "batch": 16},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["field2d", "field2d", "field2d", "field2d", "sweep", "field3d", "field3d", "leap", "train"])
    if kind == "field2d":
        nx, ny = _log_uniform(rng, 24, 6000), _log_uniform(rng, 24, 6000)
        if rng.random() < 0.6:
            nx = max(4, nx // 4 * 4)
        steps = rng.choice([1, 2, 5, 20, 50, 100])
        while steps > 1 and steps * nx * ny > 20 * 6000 * 6000:
            steps //= 2
        return {"kind": kind, "nx": nx, "ny": ny, "storage": rng.choice(["f32", "f32", "bf16", "f16"]), "steps": steps,
                "ic": rng.choice(["droplet", "spinodal"]), "alpha": round(rng.uniform(0.0, 0.5), 3), "log": False,
                "rates": "other" if rng.random() < 0.15 else "default"}
    if kind == "sweep":
        edges = rng.choice(["64,128,256,512", "64,96,128,200", "48,100,250,320", "33,65,130,257"])
        return {"kind": kind, "count": _log_uniform(rng, 16, 256), "edges": edges, "storage": rng.choice(["f32", "bf16"]),
                "steps": rng.choice([10, 50, 64]), "spec": rng.randrange(1000)}
    if kind == "field3d":
        n = [_log_uniform(rng, 16, 200) for _ in range(3)]
        return {"kind": kind, "nx": n[0], "ny": n[1], "nz": n[2], "steps": rng.choice([10, 50, 200]),
                "ic": rng.choice(["droplet", "spinodal"]), "alpha": round(rng.uniform(0.0, 0.5), 3)}
    if kind == "leap":
        return {"kind": kind, "n": rng.choice([256, 384, 512, 640]), "turns": rng.choice([1, 4]),
                "cycles": rng.choice([1, 2]), "corr": rng.choice([20, 50]), "alpha": round(rng.uniform(0.1, 0.45), 3)}
    return {"kind": kind, "n": rng.choice([128, 256, 384, 512]), "batch": rng.randint(2, 16)}


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 31))


def _field(shape, ic, seed, radius=None):
    """A seeded initial field on the GPU: U[-0.05, 0.05] noise, or a droplet (tanh profile of
    width sqrt(2) 1.5, radius 0.3 of the shortest edge) whose centre the seed moves. FP32."""
    g = _gen(seed)
    if ic == "spinodal":
        return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32) * 0.1 - 0.05
    off = torch.rand(len(shape) + 1, generator=g, device="cuda", dtype=torch.float64)
    r2 = torch.zeros(shape, device="cuda", dtype=torch.float64)
    for d, n in enumerate(shape):
        x = torch.arange(n, device="cuda", dtype=torch.float64) - n / 2.0 - (off[d] - 0.5)
        r2 += (x * x).reshape([-1 if k == d else 1 for k in range(len(shape))])
    rad = (0.28 + 0.04 * off[-1]) * min(shape)
    return torch.tanh((rad - r2.sqrt()) / (math.sqrt(2.0) * 1.5)).float()


def _sweep_specs(case):
    """Edge, strength, initial field and seed offset of each field of a sweep."""
    r = np.random.default_rng(case["spec"])
    edges = np.array([int(v) for v in case["edges"].split(",")])
    n = r.choice(edges, size=case["count"])
    alpha = r.uniform(0.0, 0.5, size=case["count"])
    return [(int(n[i]), float(alpha[i]), "droplet" if i % 2 == 0 else "spinodal", 1 + i) for i in range(case["count"])]


def _pairs(case, seed):
    """Field pairs for a training step: band-limited random fields with phases near +-1 (the
    look of a coarsening field), and the same fields moved on a little."""
    g, n, b = _gen(seed), case["n"], case["batch"]
    k = 2.0 * math.pi * torch.fft.fftfreq(n, device="cuda", dtype=torch.float64)
    q = torch.sqrt(k[:, None] ** 2 + k[None, :] ** 2)

    def band(q0):
        white = torch.randn((b, n, n), generator=g, device="cuda", dtype=torch.float64)
        v = torch.fft.ifft2(torch.fft.fft2(white) * torch.exp(-((q - q0) / 0.08) ** 2)).real
        return v / v.std(dim=(1, 2), keepdim=True)

    x = torch.tanh(0.6 * band(0.28))
    y = x + 0.01 * band(0.24)
    alpha = np.linspace(0.05, 0.5, b)
    x, y = x.float(), y.float()
    weight = 1.0 / ((y - x) ** 2).mean(dim=(1, 2)).double().cpu().numpy()
    return x.contiguous(), y.contiguous(), alpha, weight


def prepare(case, seed):
    kind = case["kind"]
    if kind == "field2d":
        kw = {"s": OTHER_RATES} if case["rates"] == "other" else {}
        s = lbch.Solver(lbch.make_params(case["nx"], case["ny"], alpha=case["alpha"], storage=STORAGE[case["storage"]], **kw))
        s.init_field_device(_field((case["ny"], case["nx"]), case["ic"], seed))
        out = torch.empty((case["ny"], case["nx"]), dtype=torch.float32, device="cuda")
        return {"kind": kind, "solver": s, "steps": case["steps"], "log": case["log"], "out": out}
    if kind == "field3d":
        s = lbch.Solver3(lbch.make_params3(case["nx"], case["ny"], case["nz"], alpha=case["alpha"]))
        s.init_field(_field((case["nz"], case["ny"], case["nx"]), case["ic"], seed).double().cpu().numpy())
        return {"kind": kind, "solver": s, "steps": case["steps"]}
    if kind == "sweep":
        specs = _sweep_specs(case)
        sizes = [n for n, _, _, _ in specs]
        b = lbch.Batch(lbch.make_params(8, 8, storage=STORAGE[case["storage"]]), sizes, sizes, [a for _, a, _, _ in specs])
        for i, (n, _, ic, k) in enumerate(specs):
            b.init_field(i, _field((n, n), ic, seed * 1009 + k).double().cpu().numpy())
        out = torch.empty(sum(n * n for n in sizes), dtype=torch.float32, device="cuda")
        return {"kind": kind, "batch": b, "steps": case["steps"], "out": out,
                "views": torch.split(out, [n * n for n in sizes])}
    if kind == "leap":
        n = case["n"]
        net = lbnop.Surrogate(n, n, max_batch=case["turns"], scale=LEAP_SCALE)
        net.set_params(np.load(WEIGHTS))
        net.set_leap_turns(case["turns"])
        s = lbch.Solver(lbch.make_params(n, n, alpha=case["alpha"]), stream=net.stream)
        s.init_field_device(_field((n, n), "spinodal", seed))
        s.step(LEAP_WARMUP)
        return {"kind": kind, "net": net, "solver": s, "alpha": case["alpha"], "cycles": case["cycles"],
                "corr": case["corr"], "judge": lbnop.make_judge(leap_steps=LEAP_STEPS), "start": s.phi_device(),
                "out": torch.empty((n, n), dtype=torch.float32, device="cuda")}
    x, y, alpha, weight = _pairs(case, seed)
    net = lbnop.Surrogate(case["n"], case["n"], max_batch=case["batch"], scale=LEAP_SCALE)
    net.set_params(np.load(WEIGHTS))
    return {"kind": kind, "net": net, "x": x, "y": y, "alpha": alpha, "weight": weight}


def run(state):
    kind = state["kind"]
    if kind == "field2d":
        s = state["solver"]
        s.step(state["steps"])
        got = {"phi": s.phi_device(state["out"])}
        if state["log"]:
            got["mass"], got["energy"] = s.mass(), s.free_energy()
        return got
    if kind == "field3d":
        s = state["solver"]
        s.step(state["steps"])
        return {"phi": s.field().astype(np.float32)}  # a snapshot at the precision that is computed
    if kind == "sweep":
        b = state["batch"]
        b.step(state["steps"])
        for i, v in enumerate(state["views"]):
            b.phi_device(i, v)
        return {"phi": state["out"]}
    if kind == "leap":  # a run from a snapshot
        state["solver"].init_field_device(state["start"])
        st = state["net"].leap_run_judged(state["solver"], state["alpha"], state["cycles"], state["corr"], state["judge"])
        return {"phi": state["solver"].phi_device(state["out"]), "accepted": st["accepted"], "rejected": st["rejected"]}
    net = state["net"]
    net.train_step(state["x"], state["alpha"], state["y"], LR, weight=state["weight"])
    return {"grad_norm": net.grad_norm(), "theta": net.params_host()}


# ---------------------------------------------------------------- what a pass cannot do without

# FP32 operations of one node update, counted from the scheme's formulas (stencils, normal and
# anisotropy, chemical potentials, relaxation with its forcing).
FLOPS_2D, FLOPS_3D = 230, 420
NET = [(16, 96, 0), (96, 96, 0), (96, 64, 1), (64, 64, 1), (64, 96, 2), (96, 96, 2), (96, 96, 3), (96, 96, 3),
       (96, 96, 2), (96, 64, 2), (64, 64, 1), (64, 96, 1), (96, 96, 0), (96, 16, 0), (16, 16, 0), (16, 16, 0)]


def _net_flops(n):
    return sum(2 * 9 * ci * co * ((n // 4) >> lv) ** 2 for ci, co, lv in NET)


def work(case):
    kind = case["kind"]
    if kind == "field2d":
        n = case["nx"] * case["ny"]
        return {"bytes": n * ((72 if case["storage"] == "f32" else 48) + 4), "flops": n * case["steps"] * FLOPS_2D}
    if kind == "field3d":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": n * (120 + 4), "flops": n * case["steps"] * FLOPS_3D}
    if kind == "sweep":
        n = sum(e * e for e, _, _, _ in _sweep_specs(case))
        return {"bytes": n * ((72 if case["storage"] == "f32" else 48) + 4), "flops": n * case["steps"] * FLOPS_2D}
    params = 4 * sum(9 * ci * co + co for ci, co, _ in NET)
    if kind == "leap":
        n = case["n"] ** 2
        return {"bytes": n * (72 + 4) + params,
                "flops": case["cycles"] * (case["turns"] * _net_flops(case["n"]) + n * case["corr"] * FLOPS_2D)}
    return {"bytes": case["batch"] * case["n"] ** 2 * 8 + 6 * params, "flops": 3 * case["batch"] * _net_flops(case["n"])}


# ---------------------------------------------------------------- the same in 64 bits

C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 1), (-1, -1, -1),
      (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (1, -1, -1), (-1, 1, 1)]
W3 = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8


def _at(a, c):
    """The field whose value at x is a(x + c), periodic in the last len(c) axes (x last)."""
    dims = [-1 - d for d in range(len(c)) if c[d]]
    return torch.roll(a, [-c[-1 - d] for d in dims], dims) if dims else a


def _grad_lap(a, C, W):
    d = len(C[0])
    g, lap = [0.0] * d, 0.0
    for c, w in zip(C[1:], W[1:]):
        v = _at(a, c)
        lap = lap + 6.0 * w * (v - a)
        for k in range(d):
            if c[k]:
                g[k] = g[k] + 3.0 * w * c[k] * v
    return g, lap


def _moments_2d():
    c = torch.tensor(C2, dtype=torch.float64)
    x, y = c[:, 0], c[:, 1]
    r = x * x + y * y
    return torch.stack([torch.ones(9, dtype=torch.float64), 3 * r - 4, 4 - 10.5 * r + 4.5 * r * r, x, (3 * r - 5) * x, y,
                        (3 * r - 5) * y, x * x - y * y, x * y])


def _scheme(phi0, alpha, steps, C, W, rates=None):
    """phi after `steps` time steps from f = f^eq(phi0), mass and free energy; FP64."""
    d, q = len(C[0]), len(C)
    beta, k = 3 * SIGMA / (4 * DW), 3 * SIGMA * DW / 8
    sj = 1.0 / (3.0 * M + 0.5)

    def fields(phi):
        g, lap = _grad_lap(phi, C, W)
        g2 = sum(v * v for v in g)
        ok = g2 >= 1e-12
        nrm = g2.sqrt()
        n = [torch.where(ok, v / torch.where(ok, nrm, 1.0), 0.0) for v in g]
        s4 = sum(v ** 4 for v in n)
        gm1 = torch.where(ok, alpha * (4.0 * s4 - 3.0), 0.0)
        fb = 4 * beta * phi * (phi * phi - 1.0)
        return g, g2, lap, nrm, n, s4, gm1, fb

    def collide(f, phi):
        g, _, lap, nrm, n, s4, gm1, fb = fields(phi)
        mua = fb - k * lap
        w = lap - fb
        mub = gm1 * fb + EPS * (_grad_lap(w, C, W)[1] - 4 * beta * (3 * phi * phi - 1.0) * w)
        for a in range(d):
            Q = gm1 * k * g[a] + k * nrm * 16.0 * alpha * n[a] * (n[a] * n[a] - s4)
            mub = mub - _grad_lap(Q, C, W)[0][a]
        del g, n, lap, w, Q
        gb = _grad_lap(mub, C, W)[0]
        if rates is None:  # every moment but phi and the flux relaxes fully: f* in closed form
            j = [sum(c[a] * f[i] for i, c in enumerate(C) if c[a]) for a in range(d)]
            for i in range(1, q):
                # f^eq + F/2, and the flux's own rate: its projection w_i c.(.) / (1/3)
                v = mua + sum(c_a * (-0.5 * gb_a) for c_a, gb_a in zip(C[i], gb) if c_a)
                jn = sum(c_a * ((1 - sj) * j_a + (0.5 - 0.5 * sj) * (-gb_a / 3.0)) for c_a, j_a, gb_a in zip(C[i], j, gb) if c_a)
                c2 = sum(c_a * c_a for c_a in C[i])
                f[i] = W[i] * v + jn * JW[d][c2]
            f[0] = phi - f[1:].sum(dim=0)
        else:
            feq = torch.stack([w_i * mua for w_i in W])
            feq[0] += phi - mua
            F = torch.stack([-w_i * (c[0] * gb[0] + c[1] * gb[1]) for c, w_i in zip(C, W)])
            mm = _moments_2d()
            s = torch.tensor(rates, dtype=torch.float64)
            s[3] = s[5] = sj
            mi = torch.linalg.inv(mm)
            A = (mi @ torch.diag(s) @ mm).to(f.device)
            B = (mi @ torch.diag(1.0 - s / 2.0) @ mm).to(f.device)
            f -= torch.tensordot(A, f - feq, 1)
            f += torch.tensordot(B, F, 1)
        for i in range(1, q):
            f[i] = _at(f[i], tuple(-v for v in C[i]))
        return f

    # weight of the flux j in population i of M^-1 (the j rows have squared norms 6 and 10)
    JW = {2: {1: 1 / 6, 2: 1 / 6}, 3: {1: 1 / 10, 2: 0.0, 3: 1 / 10}}
    lap0 = _grad_lap(phi0, C, W)[1]
    mua = 4 * beta * phi0 * (phi0 * phi0 - 1.0) - k * lap0
    f = torch.stack([w_i * mua for w_i in W])
    f[0] += phi0 - mua
    del lap0, mua
    for _ in range(steps):
        f = collide(f, f.sum(dim=0))
    phi = f.sum(dim=0)
    del f
    _, g2, lap, _, _, _, gm1, fb = fields(phi)
    e = (1.0 + gm1) * (0.5 * k * g2 + beta * (phi * phi - 1.0) ** 2) + 0.5 * EPS * (lap - fb) ** 2
    return phi, float(phi.sum()), float(e.sum())


def _net_layers(theta):
    out, at = [], 0
    for k, (ci, co, _) in enumerate(NET):
        w = theta[at:at + 9 * ci * co].reshape(3, 3, co, ci).permute(2, 3, 0, 1)
        at += 9 * ci * co
        b = theta[at:at + co]
        at += co
        v = None
        if k == 0:
            v = theta[at:at + co]
            at += co
        out.append((w, b, v))
    return out


def _net(theta, phi, alpha):
    """phi(t + K) of the leap network for phi [B][H][W], alpha [B]; FP64."""
    F = torch.nn.functional
    P = _net_layers(theta)
    al = alpha.reshape(-1, 1, 1, 1)

    def conv(k, x):
        z = F.conv2d(F.pad(x, (1, 1, 1, 1), mode="circular"), P[k][0], P[k][1])
        return z + al * P[k][2].reshape(1, -1, 1, 1) if k == 0 else z

    def up(x):
        return F.interpolate(x, scale_factor=2, mode="nearest")

    act, pool = F.silu, lambda x: F.avg_pool2d(x, 2)  # noqa: E731
    sig = (phi * phi).mean(dim=(1, 2), keepdim=True).sqrt()
    x0 = F.pixel_unshuffle((phi / sig).unsqueeze(1), 4)
    h0 = act(conv(1, act(conv(0, x0))))
    h1 = act(conv(3, act(conv(2, pool(h0)))))
    h2 = act(conv(5, act(conv(4, pool(h1)))))
    h3 = act(conv(7, act(conv(6, pool(h2)))))
    z2 = conv(9, act(conv(8, up(h3) + h2)))
    z1 = conv(11, act(conv(10, up(z2) + h1)))
    zo = conv(13, act(conv(12, up(z1) + h0))) + conv(14, x0) + al * conv(15, x0)
    D = F.pixel_shuffle(zo, 4).squeeze(1)
    return phi + LEAP_SCALE * sig * (D - D.mean(dim=(1, 2), keepdim=True))


def exact(case, seed):
    kind = case["kind"]
    if kind == "field2d":
        if case["nx"] * case["ny"] * case["steps"] > 3e9:
            return None
        phi0 = _field((case["ny"], case["nx"]), case["ic"], seed).double()
        phi, mass, energy = _scheme(phi0, case["alpha"], case["steps"], C2, W2, OTHER_RATES if case["rates"] == "other" else None)
        return {"phi": phi, "mass": mass, "energy": energy} if case["log"] else {"phi": phi}
    if kind == "field3d":
        phi0 = _field((case["nz"], case["ny"], case["nx"]), case["ic"], seed).double()
        return {"phi": _scheme(phi0, case["alpha"], case["steps"], C3, W3)[0]}
    if kind == "sweep":
        specs = _sweep_specs(case)
        got = [None] * len(specs)
        for n in sorted({s[0] for s in specs}):
            ids = [i for i, s in enumerate(specs) if s[0] == n]
            phi0 = torch.stack([_field((n, n), specs[i][2], seed * 1009 + specs[i][3]) for i in ids]).double()
            al = torch.tensor([specs[i][1] for i in ids], dtype=torch.float64, device="cuda").reshape(-1, 1, 1)
            phi = _scheme(phi0, al, case["steps"], C2, W2)[0]
            for k, i in enumerate(ids):
                got[i] = phi[k].reshape(-1)
        return {"phi": torch.cat(got)}
    theta = torch.from_numpy(np.load(WEIGHTS)).cuda().double()
    if kind == "leap":
        n, al = case["n"], torch.tensor([case["alpha"]], dtype=torch.float64, device="cuda")
        phi = _scheme(_field((n, n), "spinodal", seed).double(), case["alpha"], LEAP_WARMUP, C2, W2)[0]
        with torch.no_grad():
            for _ in range(case["cycles"]):
                turns = range(0, 4) if case["turns"] == 4 else [0]
                phi = torch.stack([torch.rot90(_net(theta, torch.rot90(phi[None], t, dims=(1, 2)), al), -t, dims=(1, 2))[0]
                                   for t in turns]).mean(dim=0)
                phi = _scheme(phi, case["alpha"], case["corr"], C2, W2)[0]
        return {"phi": phi, "accepted": None, "rejected": None}
    x, y, alpha, weight = _pairs(case, seed)
    theta.requires_grad_(True)
    al = torch.from_numpy(alpha).cuda()
    w = torch.from_numpy(weight).cuda().reshape(-1, 1, 1)
    for b in range(case["batch"]):  # one sample at a time: FP64 activations are large
        out = _net(theta, x[b:b + 1].double(), al[b:b + 1])
        (w[b:b + 1] * (out - y[b:b + 1].double()) ** 2).sum().div(x.numel()).backward()
    g = theta.grad
    new = theta.detach() - LR * g / (g.abs() + 1e-8)  # Adam's first step
    return {"grad_norm": float(g.norm()), "theta": new}
