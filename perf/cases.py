"""What a user of this framework has it do, as timed cases.

Five kinds of work, each through the public Python entry points:

  lattice   one lattice: initialise from (P, u), advance, read the derived
            fields (Lattice.init / set_force / step / step_fields / fields);
  cavities  a batch of lid-driven cavities advanced with convergence checks
            and read back (CavityBatch.init / run / fields_host);
  unet      the warm-start network: inference, or the loss and gradients of
            one minibatch (WarmStartNet.forward / train_step / get_params);
  conv      one convolution layer of that network, forward;
  convback  the backward pass of one such layer.

`listed()` are the measured cases, `draw(rng)` makes more of the same ranges,
`prepare` makes what a program holds before the call, `run` is one pass,
`work` its unavoidable bytes and operations, `exact` its result in 64 bits
from plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2108_08591_gb300 import (CavityBatch, Lattice, WarmStartNet, conv3x3_bf16,
                                    conv3x3_bf16_backward)

POP_BYTES = {"f32": 4, "f16": 2, "bf16": 2, "f64": 8, "f16eq": 2, "bf16eq": 2}
ALL_FIELDS = ("P", "u", "G", "S", "sigma", "omega")  # div is identically zero (Eq. 3-16a)


def _lat(name, shape, storage, steps, bc="periodic", force=False, scheme2=False, inplace=False, q=0,
         epilogue=False, fields="P,u,G,S,omega"):
    c = {"kind": "lattice", "shape": "x".join(str(n) for n in shape), "storage": storage,
         "steps": steps, "bc": bc, "force": force, "scheme2": scheme2, "inplace": inplace, "q": q,
         "epilogue": epilogue, "fields": fields}
    if name:
        c["name"] = name
    return c


def _named(name, **kw):
    return dict(kw, name=name) if name else kw


def listed():
    return [
        # the four-roll mill of the paper's Table 1: a 64^2 box with a body force,
        # as in any convergence study; latency and launches count
        _lat("mill2d_64_f32", (64, 64), "f32", 100, force=True),
        # the headline 2D run: one epilogue period (fields every 50 updates here)
        _lat("tg2d_4096_f32", (4096, 4096), "f32", 100, epilogue=True),
        # a lid-driven cavity of odd sides (the paper's Table 2 size, off the powers of two)
        _lat("cavity2d_509x515_f32", (509, 515), "f32", 100, bc="cavity"),
        # reduced-precision storage in 2D, sides that are no power of two
        _lat("tg2d_2050x1998_f16eq", (2050, 1998), "f16eq", 60),
        # 3D Taylor-Green vortex, FP32
        _lat("tg3d_256_f32", (256, 256, 256), "f32", 40, fields="P,u"),
        # 3D with reduced-precision storage, a ragged box
        _lat("tg3d_190x202x178_bf16eq", (190, 202, 178), "bf16eq", 40),
        # a few small cavities: a Reynolds-number sweep at the paper's scale
        _named("cavities_12_small", kind="cavities", sides="65,65,65,97,97,97,97,97,129,129,129,129",
               steps=1000, seed_re=7),
        # the mixed batch: sides 65 .. 513, larger than L2
        _named("cavities_28_mixed", kind="cavities",
               sides=",".join(["65"] * 5 + ["129"] * 7 + ["257"] * 7 + ["513"] * 9),
               steps=1000, seed_re=2108),
        # network inference for a batch of 256^2 cavities
        _named("unet_forward_256_b8", kind="unet", side=256, batch=8, channels="32,64,128,256", grad=False),
        # loss and gradients of one minibatch
        _named("unet_gradient_256_b8", kind="unet", side=256, batch=8, channels="32,64,128,256", grad=True),
        # the widest full-resolution layer of the network, forward with bias and ReLU
        _named("conv_8x256x256_96to32", kind="conv", B=8, H=256, W=256, Cin=96, Cout=32, relu=True, out_fp32=False),
        # backward of a deep layer
        _named("convback_8x64x64_128to128", kind="convback", B=8, H=64, W=64, Cin=128, Cout=128),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lat2d", "lat2d", "lat2d", "lat3d", "lat3d", "cavities", "unet", "conv", "convback"])
    if kind == "lat2d":
        storage = rng.choice(["f32", "f32", "f32", "f16eq", "bf16eq", "f16", "bf16", "f64"])
        nx, ny = _logint(rng, 24, 4096), _logint(rng, 24, 4000)
        if rng.random() < 0.5:
            nx = max(32, nx // 4 * 4)
        bc = rng.choice(["periodic", "periodic", "channel", "cavity"])
        rest_shifted = storage in ("f32", "f64", "f16", "bf16")
        force = bc == "channel" or rng.random() < 0.25
        return _lat(None, (nx, ny), storage, rng.choice([1, 3, 10, 25, 50]), bc=bc, force=force,
                    scheme2=force and rng.random() < 0.4, inplace=rest_shifted and rng.random() < 0.2,
                    q=4 if rest_shifted and rng.random() < 0.15 else 0, epilogue=rng.random() < 0.3,
                    fields=rng.choice(["P,u", "P,u,G,S,omega"]))
    if kind == "lat3d":
        storage = rng.choice(["f32", "f32", "f16eq", "bf16eq", "f16"])
        shape = [_logint(rng, 16, 256) for _ in range(3)]
        if rng.random() < 0.5:
            shape[0] = max(16, shape[0] // 4 * 4)
        bc = rng.choice(["periodic", "periodic", "channel", "cavity"])
        rest_shifted = storage in ("f32", "f16")
        force = bc == "channel"
        return _lat(None, shape, storage, rng.choice([1, 4, 15, 40]), bc=bc, force=force,
                    inplace=rest_shifted and rng.random() < 0.2,
                    q=6 if rest_shifted and rng.random() < 0.15 else 0,
                    fields=rng.choice(["P,u", "P,u,G,S,omega"]))
    if kind == "cavities":
        kinds = [_logint(rng, 33, 400) for _ in range(rng.randint(1, 3))]
        n = _logint(rng, 2, 28)
        return {"kind": "cavities", "sides": ",".join(str(rng.choice(kinds)) for _ in range(n)),
                "steps": rng.choice([200, 400]), "seed_re": rng.randint(1, 10 ** 6)}
    if kind == "unet":
        return {"kind": "unet", "side": rng.choice([64, 96, 128, 192, 256]), "batch": rng.randint(1, 8),
                "channels": rng.choice(["16,32,64", "32,64,128", "32,64,128,256"]), "grad": rng.random() < 0.5}
    B, H, W = rng.randint(1, 8), _logint(rng, 16, 256), _logint(rng, 16, 256)
    cin, cout = 16 * rng.randint(1, 12), 16 * rng.randint(1, 12)
    while B * H * W * cin * cout > 8 * 256 * 256 * 96 * 32:
        cin, cout = max(16, cin // 32 * 16), max(16, cout // 32 * 16)
    if kind == "conv":
        return {"kind": "conv", "B": B, "H": H, "W": W, "Cin": cin, "Cout": cout,
                "relu": rng.random() < 0.7, "out_fp32": rng.random() < 0.3}
    return {"kind": "convback", "B": B, "H": H, "W": W, "Cin": cin, "Cout": cout}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _rates(case):
    """(s1, s2): nu = 0.01 and the paper's s2 rule in 2D; the 3D Taylor-Green
    rates (s1 = 1.96, s2 = 1) in 3D."""
    if len(_shape(case)) == 2:
        cs2 = 0.5 if case["q"] == 4 else 1.0 / 3.0
        s1 = 1.0 / (0.01 / cs2 + 0.5)
        return s1, 8.0 * (2.0 - s1) / (8.0 - s1)
    cs2 = 1.0 / 3.0 if case["q"] == 6 else 0.25
    return 1.0 / (0.0026 / cs2 + 0.5), 1.0


def _walls(case):
    """(wall per axis, lid, lid velocity)."""
    d = len(_shape(case))
    if case["bc"] == "channel":
        return (0,) * (d - 1) + (1,), False, (0.0, 0.0, 0.0)
    if case["bc"] == "cavity":
        return (1,) * d, True, (0.1, 0.0, 0.0)
    return (0,) * d, False, (0.0, 0.0, 0.0)


def _flow(case, seed):
    """Seeded start (P [N], u [d][N]) and force (or None), FP64 on the GPU: a
    Taylor-Green vortex plus a few low divergence-free modes, x fastest."""
    shape = _shape(case)
    d = len(shape)
    rng = np.random.default_rng([seed, *shape])
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n) for n in shape]
    X = ax[0].view((1,) * (d - 1) + (-1,))
    Y = ax[1].view((1,) * (d - 2) + (-1, 1))
    Z = ax[2].view(-1, 1, 1) if d == 3 else torch.zeros((1, 1), dtype=torch.float64, device="cuda")
    U0 = 0.01 if d == 2 else 0.05
    px, py = rng.uniform(0, 2 * math.pi, 2)
    zc = torch.cos(Z) if d == 3 else 1.0
    full = torch.zeros(shape[::-1], dtype=torch.float64, device="cuda")
    # stretch the second component so that the field stays divergence-free
    ry = shape[1] / shape[0]
    u = [U0 * torch.sin(X + px) * torch.cos(Y + py) * zc + full,
         -U0 * ry * torch.cos(X + px) * torch.sin(Y + py) * zc + full]
    P = 1.0 + 0.25 * U0 * U0 * (torch.cos(2 * (X + px)) + torch.cos(2 * (Y + py))) * (zc * zc) + full
    for _ in range(4):
        mx, my = int(rng.integers(1, 5)), int(rng.integers(1, 5))
        ph, amp = rng.uniform(0, 2 * math.pi), U0 * rng.uniform(0.05, 0.15)
        s = torch.sin(mx * X + my * Y + ph)
        n = math.hypot(mx / shape[0], my / shape[1])
        u[0] += amp * (my / shape[1]) / n * s
        u[1] -= amp * (mx / shape[0]) / n * s
    if d == 3:
        u.append(0.1 * U0 * torch.sin(X + Y + px) + full)
    F = None
    if case["force"]:
        F = torch.zeros((d, *shape[::-1]), dtype=torch.float64, device="cuda")
        if case["bc"] == "channel":
            F[0] += 1e-6 * rng.uniform(0.5, 1.5)
        else:
            f0 = 1e-6 * rng.uniform(0.5, 1.5)
            F[0] += f0 * torch.sin(X) * torch.cos(Y)
            F[1] -= f0 * torch.cos(X) * torch.sin(Y)
        F = F.reshape(d, -1).contiguous()
    return P.reshape(-1).contiguous(), torch.stack(u).reshape(d, -1).contiguous(), F


def _sides(case):
    return [int(s) for s in case["sides"].split(",")]


def _reynolds(case, seed):
    rng = np.random.default_rng([seed, case["seed_re"]])
    return [float(rng.uniform(60.0, min(1000.0, 4.0 * s))) for s in _sides(case)]


def _net_batch(case, seed):
    """Input planes (Re, lid speed, node coordinates, lid row, wall rows) and
    smooth targets of a minibatch of cavities."""
    n, B = case["side"], case["batch"]
    rng = np.random.default_rng([seed, n, B])
    c = (torch.arange(n, dtype=torch.float32, device="cuda") + 0.5) / n
    x = torch.zeros((B, n, n, 16), dtype=torch.float32, device="cuda")
    x[..., 0] = torch.tensor(rng.uniform(0.1, 1.0, B), dtype=torch.float32, device="cuda").view(B, 1, 1)
    x[..., 1] = 1.0
    x[..., 2] = c.view(1, 1, n)
    x[..., 3] = c.view(1, n, 1)
    x[:, n - 1, :, 4] = 1.0
    x[:, 0, :, 5] = x[:, n - 1, :, 5] = 1.0
    x[:, :, 0, 5] = x[:, :, n - 1, 5] = 1.0
    t = torch.stack([torch.sin(3 * x[..., 2] + k) * torch.cos(2 * x[..., 3]) * x[..., 0] for k in range(3)], -1)
    return x, t.contiguous()


def _net_params(case, seed):
    """He-uniform weights [Cout][3][3][Cin] and small biases of every convolution, flat."""
    rng = np.random.default_rng([seed, 3, case["side"]])
    parts = []
    for _, ci, co in _net_layers(case):
        parts.append(rng.uniform(-1.0, 1.0, co * 9 * ci) * math.sqrt(6.0 / (9 * ci)))
        parts.append(rng.uniform(-0.05, 0.05, co))
    return np.concatenate(parts).astype(np.float32)


def _layer(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed * 1000003 + case["Cin"] * 131 + case["Cout"])
    B, H, W, ci, co = (case[k] for k in ("B", "H", "W", "Cin", "Cout"))
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float32)
    # activations after a ReLU, He-scaled weights
    x = torch.relu(rnd(B, H, W, ci)).to(torch.bfloat16)
    w = (rnd(co, 3, 3, ci) * math.sqrt(2.0 / (9 * ci))).to(torch.bfloat16)
    return x, w, rnd(co) * 0.1, (rnd(B, H, W, co) * 0.01).to(torch.bfloat16)


# ---------------------------------------------------------------------------
# Measured passes
# ---------------------------------------------------------------------------
def prepare(case, seed):
    k = case["kind"]
    if k == "lattice":
        P, u, F = _flow(case, seed)
        s1, s2 = _rates(case)
        wall, lid, lid_u = _walls(case)
        lat = Lattice(_shape(case), s1, s2=s2, wall=wall, lid=lid, lid_u=lid_u, storage=case["storage"],
                      q=case["q"], inplace=case["inplace"])
        if case["scheme2"]:
            lat.set_forcing("scheme2")
        if F is not None:
            lat.set_force(F)
        return {"case": case, "lat": lat, "P": P, "u": u}
    if k == "cavities":
        return {"case": case, "batch": CavityBatch(_sides(case), _reynolds(case, seed), lid_speed=0.1)}
    if k == "unet":
        x, t = _net_batch(case, seed)
        net = WarmStartNet(case["side"], case["side"], [int(c) for c in case["channels"].split(",")],
                           max_batch=case["batch"])
        net.set_params(_net_params(case, seed))
        return {"case": case, "net": net, "x": x, "t": t}
    x, w, bias, dz = _layer(case, seed)
    return {"case": case, "x": x, "w": w, "bias": bias, "dz": dz}


def run(state):
    case = state["case"]
    k = case["kind"]
    if k == "lattice":
        lat, n = state["lat"], case["steps"]
        lat.init(state["P"], state["u"])
        names = case["fields"].split(",")
        mid = {}
        if case["epilogue"]:  # fields of the state half way, written by the update itself
            half = n // 2
            lat.step(half)
            mid = lat.alloc_fields(ALL_FIELDS)
            lat.step_fields(n - half, mid)
        else:
            lat.step(n)
        return {**{"mid_" + f: v for f, v in mid.items()}, **lat.fields(names)}
    if k == "cavities":
        b = state["batch"]
        b.init()
        steps, status, res = b.run(tol=1e-8, max_steps=case["steps"], check_every=100)
        return {"steps": steps, "status": status, "residual": res,
                "fields": [b.fields_host(c) for c in range(b.n)]}
    if k == "unet":
        net = state["net"]
        if not case["grad"]:
            return net.forward(state["x"])
        loss = net.train_step(state["x"], state["t"], 0.0)
        return {"loss": loss, "grads": net.get_params(grads=True)[1]}
    if k == "conv":
        return conv3x3_bf16(state["x"], state["w"], state["bias"], relu=case["relu"], out_fp32=case["out_fp32"])
    return conv3x3_bf16_backward(state["x"], state["w"], state["dz"])


# ---------------------------------------------------------------------------
# Unavoidable work
# ---------------------------------------------------------------------------
def _net_layers(case):
    """(side, Cin, Cout) of every convolution, in the network's order."""
    C, n = [int(c) for c in case["channels"].split(",")], case["side"]
    out, c = [], 16
    for l, ch in enumerate(C):
        out += [(n >> l, c, ch), (n >> l, ch, ch)]
        c = ch
    for l in range(len(C) - 2, -1, -1):
        out += [(n >> l, C[l + 1] + C[l], C[l]), (n >> l, C[l], C[l])]
    return out + [(n, C[0], 16)]


def work(case):
    k = case["kind"]
    if k == "lattice":
        shape = _shape(case)
        d, N = len(shape), math.prod(shape)
        q = case["q"] or (5 if d == 2 else 7)
        count = {"P": 1, "u": d, "G": d * d, "div": 1, "S": 3 if d == 2 else 6, "sigma": 3 if d == 2 else 6,
                 "omega": 1 if d == 2 else 3}
        out = sum(count[f] for f in case["fields"].split(","))
        if case["epilogue"]:
            out += sum(count.values())
        # P and u in, the fields out, and the state once in memory; per node and
        # update and set: moments, equilibrium, relaxation, ~10 operations per direction
        state = q * (d + 1) * POP_BYTES[case["storage"]]
        return {"bytes": N * (8 * (1 + d) + 8 * out + 2 * state),
                "flops": N * case["steps"] * (d + 1) * q * 10}
    if k == "cavities":
        N = sum(s * s for s in _sides(case))
        return {"bytes": N * (2 * 60 + 24), "flops": N * case["steps"] * 150}
    if k == "unet":
        B = case["batch"]
        layers = _net_layers(case)
        fl = sum(2 * B * s * s * ci * 9 * co for s, ci, co in layers)
        by = sum(2 * B * s * s * (ci + co) + 18 * ci * co for s, ci, co in layers)
        return {"bytes": by * (3 if case["grad"] else 1), "flops": fl * (3 if case["grad"] else 1)}
    B, H, W, ci, co = (case[x] for x in ("B", "H", "W", "Cin", "Cout"))
    M = B * H * W
    fl = 2 * M * ci * 9 * co
    if k == "conv":
        return {"bytes": 2 * M * ci + 18 * ci * co + M * co * (4 if case["out_fp32"] else 2), "flops": fl}
    return {"bytes": 2 * M * (2 * ci + co) + 18 * ci * co + 36 * ci * co, "flops": 2 * fl}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
# velocities as the axis and sign of each direction (None: rest), weights, c_s^2
_LATTICES = {
    4: ([(0, 1), (1, 1), (0, -1), (1, -1)], [0.25] * 4, 0.5),
    5: ([None, (0, 1), (1, 1), (0, -1), (1, -1)], [1 / 3] + [1 / 6] * 4, 1 / 3),
    6: ([(0, 1), (0, -1), (1, 1), (1, -1), (2, 1), (2, -1)], [1 / 6] * 6, 1 / 3),
    7: ([None, (0, 1), (0, -1), (1, 1), (1, -1), (2, 1), (2, -1)], [0.25] + [0.125] * 6, 0.25),
}


class _Ref:
    """MDF-LBM in FP64 on arrays [sets][q][...][z][y][x] (shifted by the rest
    state), advanced by the paper's update with a dense collision matrix.
    `lead` counts leading batch axes; s1, s2 may vary along them."""

    def __init__(self, d, q, s1, s2, wall, lid, lid_u, F=None, scheme2=False):
        self.d, self.q = d, q
        self.c, self.w, self.cs2 = _LATTICES[q]
        self.s1, self.wall, self.lid, self.lid_u, self.F = s1, wall, lid, lid_u, F
        self.scheme2 = scheme2 and F is not None
        self.opp = [next(j for j, e in enumerate(self.c)
                         if (e is None and v is None) or (v and e and e[0] == v[0] and e[1] == -v[1]))
                    for v in self.c]
        c = np.zeros((q, d))
        for i, v in enumerate(self.c):
            if v:
                c[i, v[0]] = v[1]
        sq = c * c
        rows, rate = [np.ones(q)] + [c[:, b] for b in range(d)], [0] + [1] * d
        if d == 2:
            rows.append(sq[:, 0] - sq[:, 1])
        else:
            rows += [2 * sq[:, 0] - sq[:, 1] - sq[:, 2], sq[:, 1] - sq[:, 2]]
        if q in (5, 7):
            rows.append((q * sq.sum(1) - 2 * d))
        rate += [2] * (q - 1 - d)
        M = np.stack(rows)
        inv = np.linalg.inv(M)
        part = lambda k: torch.tensor(inv @ np.diag([float(r == k) for r in rate]) @ M,
                                      dtype=torch.float64, device="cuda")
        self.L = [part(0), part(1), part(2)]  # Lambda = L0 + s1 L1 + s2 L2 (s0 = 1)
        self.s2 = s2

    def lam(self, a):
        return sum(s * torch.einsum("ij,j...->i...", m, a) for s, m in zip((1.0, self.s1, self.s2), self.L))

    def moments(self, g):
        u = g[1:].sum(1)
        if self.scheme2:
            u = u + 0.5 * self.F
        J = [[sum(v[1] * g[1 + a, i] for i, v in enumerate(self.c) if v and v[0] == b) for b in range(self.d)]
             for a in range(self.d)]
        P = (sum(J[a][a] for a in range(self.d)) - (u * u).sum(0)) / self.d
        return u, P, J

    def geq(self, alpha, u, P, r):
        out = []
        for i, v in enumerate(self.c):
            cu = v[1] * u[v[0]] if v else 0.0
            if alpha == 0:
                out.append(self.w[i] * (r + (1.0 + r) * cu / self.cs2))
            else:
                cP = v[1] * P if v and v[0] == alpha - 1 else 0.0
                out.append(self.w[i] * (u[alpha - 1] + (cu * u[alpha - 1] + cP) / self.cs2))
        return torch.stack([o if torch.is_tensor(o) and o.shape == P.shape else o + torch.zeros_like(P)
                            for o in out])

    def start(self, P, u):
        g = torch.stack([self.geq(a, u, P, torch.zeros_like(P)) for a in range(self.d + 1)])
        if self.scheme2:
            for a in range(self.d):
                for i in range(self.q):
                    g[1 + a, i] -= 0.5 * self.w[i] * self.F[a]
        return g

    def step(self, g):
        u, P, _ = self.moments(g)
        for alpha in range(self.d + 1):
            r = g[0].sum(0) if alpha == 0 else None
            ge = self.geq(alpha, u, P, r)
            if self.F is not None and alpha >= 1:
                wF = torch.stack([w * self.F[alpha - 1] for w in self.w])
                src = wF - 0.5 * self.lam(wF) if self.scheme2 else wF
            else:
                src = 0.0
            g[alpha] += src - self.lam(g[alpha] - ge)
        out = torch.empty_like(g)
        for i, v in enumerate(self.c):
            if v is None:
                out[:, i] = g[:, i]
                continue
            ax = g.dim() - 2 - v[0]  # axis of g[:, i]: x is the last
            out[:, i] = torch.roll(g[:, i], v[1], dims=ax)
            if self.wall[v[0]]:
                n = out[:, i].shape[ax]
                row = 0 if v[1] == 1 else n - 1
                dst = out[:, i].select(ax, row)
                dst.copy_(-g[:, self.opp[i]].select(ax, row))
                if self.lid and v[0] == self.d - 1 and v[1] == -1:
                    for a in range(self.d):
                        dst[1 + a] += 2.0 * self.w[i] * self.lid_u[a]
        return out

    def fields(self, g, names):
        d, (u, P, J) = self.d, self.moments(g)
        m = [[J[a][b] - u[a] * u[b] - (P if a == b else 0.0) for b in range(d)] for a in range(d)]
        pre, sig = -self.s1 / self.cs2, -(1.0 - 0.5 * self.s1)
        up = [(a, b) for a in range(d) for b in range(a, d)]
        rot = [(1, 0)] if d == 2 else [(2, 1), (0, 2), (1, 0)]
        one = {"P": lambda: 1.0 + P, "u": lambda: u,
               "G": lambda: torch.stack([torch.stack([pre * m[a][b] for b in range(d)]) for a in range(d)]),
               "div": lambda: pre * sum(m[a][a] for a in range(d)),
               "S": lambda: torch.stack([0.5 * pre * (m[a][b] + m[b][a]) for a, b in up]),
               "sigma": lambda: torch.stack([sig * (m[a][b] + m[b][a]) for a, b in up]),
               "omega": lambda: torch.stack([pre * (m[a][b] - m[b][a]) for a, b in rot])}
        lead = {"P": 0, "div": 0, "G": 2}
        return {n: (lambda t: t.reshape(t.shape[:lead.get(n, 1)] + (-1,)))(one[n]()) for n in names}


def _exact_lattice(case, seed):
    shape = _shape(case)
    d = len(shape)
    if math.prod(shape) * case["steps"] > (2.0e9 if d == 2 else 1.0e9):
        return None
    P, u, F = _flow(case, seed)
    s1, s2 = _rates(case)
    grid = shape[::-1]
    ref = _Ref(d, case["q"] or (5 if d == 2 else 7), s1, s2, *_walls(case),
               F=None if F is None else F.reshape(d, *grid), scheme2=case["scheme2"])
    g = ref.start(P.reshape(grid) - 1.0, u.reshape(d, *grid))
    half = case["steps"] // 2
    mid = {}
    for k in range(case["steps"]):
        if case["epilogue"] and k == half:
            mid = ref.fields(g, ALL_FIELDS)
        g = ref.step(g)
    out = ref.fields(g, case["fields"].split(","))
    return {**{"mid_" + f: v for f, v in mid.items()}, **out}


def _exact_cavities(case, seed):
    sides, Re, U = _sides(case), _reynolds(case, seed), 0.1
    if sum(s * s for s in sides) * case["steps"] > 6.0e9:
        return None
    n = len(sides)
    fields, res = [None] * n, np.zeros(n)
    for side in sorted(set(sides)):
        ids = [c for c in range(n) if sides[c] == side]
        s1 = torch.tensor([1.0 / (3.0 * U * side / Re[c] + 0.5) for c in ids], dtype=torch.float64,
                          device="cuda").view(-1, 1, 1)
        ref = _Ref(2, 5, s1, 8.0 * (2.0 - s1) / (8.0 - s1), (1, 1), True, (U, 0.0))
        zero = torch.zeros((len(ids), side, side), dtype=torch.float64, device="cuda")
        g = ref.start(zero, torch.stack([zero, zero]))
        prev = None
        for k in range(case["steps"] + 1):
            if k % 100 == 0:
                u, P, _ = ref.moments(g)
                if prev is not None:
                    last = ((u - prev) ** 2).sum((0, 2, 3)).sqrt() / (100.0 * (u * u).sum((0, 2, 3)).sqrt())
                prev = u
            if k < case["steps"]:
                g = ref.step(g)
        for j, c in enumerate(ids):
            fields[c] = {"P": (1.0 + P[j]).reshape(-1).cpu().numpy(), "u": u[:, j].reshape(2, -1).cpu().numpy()}
            res[c] = float(last[j])
    return {"steps": None, "status": None, "residual": res, "fields": fields}


def _conv64(x, w, bias=None):
    return torch.nn.functional.conv2d(x, w, bias, padding=1)


def _exact_unet(case, seed):
    x, t = _net_batch(case, seed)
    C = [int(c) for c in case["channels"].split(",")]
    flat = torch.from_numpy(_net_params(case, seed)).double().cuda().requires_grad_(case["grad"])
    p, off = [], 0
    for _, ci, co in _net_layers(case):
        w = flat[off:off + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        p.append((w, flat[off + co * 9 * ci:off + co * 9 * ci + co]))
        off += co * 9 * ci + co
    it = iter(p)
    act = lambda h: torch.relu(_conv64(h, *next(it)))
    h, skips = x.double().permute(0, 3, 1, 2), []
    for l in range(len(C)):
        if l:
            h = torch.nn.functional.avg_pool2d(h, 2)
        h = act(act(h))
        skips.append(h)
    for l in range(len(C) - 2, -1, -1):
        h = act(act(torch.cat([torch.nn.functional.interpolate(h, scale_factor=2, mode="nearest"), skips[l]], 1)))
    y = _conv64(h, *next(it)).permute(0, 2, 3, 1)
    if not case["grad"]:
        return y
    loss = ((y[..., :3] - t.double()) ** 2).mean()
    loss.backward()
    return {"loss": float(loss), "grads": flat.grad.cpu().numpy()}


def exact(case, seed):
    k = case["kind"]
    if k == "lattice":
        return _exact_lattice(case, seed)
    if k == "cavities":
        return _exact_cavities(case, seed)
    if k == "unet":
        return _exact_unet(case, seed)
    x, w, bias, dz = _layer(case, seed)
    x64 = x.double().permute(0, 3, 1, 2)
    w64 = w.double().permute(0, 3, 1, 2)
    if k == "conv":
        y = _conv64(x64, w64, bias.double())
        return (torch.relu(y) if case["relu"] else y).permute(0, 2, 3, 1)
    dz64 = dz.double().permute(0, 3, 1, 2)
    dx = torch.nn.grad.conv2d_input(x64.shape, w64, dz64, padding=1)
    dw = torch.nn.grad.conv2d_weight(x64, w64.shape, dz64, padding=1)
    return dx.permute(0, 2, 3, 1), dw.permute(0, 2, 3, 1)
