"""Timed cases of the solver and its forcing network, through the Python binding of the C ABI.

Four kinds, each the call that a program of this package makes in its loop:

  rk3     dg_rk3_step on one mesh, plain or with the network's forcing in every stage
  batch   dg_batch_rk3_step on a batch of independent flows
  sample  what a run records at a sampling time: dg_project of the high-order state to the
          low order, then dg_diagnostics of both
  train   nn_train_step on one shuffled mini-batch, as the epochs of Algorithm 1 run it

States are Taylor-Green vortices with seeded large-scale modes and small per-node noise on
top, made here in torch.  ``exact`` restates the method in 64 bits in plain torch.
"""
import math

import numpy as np
import torch

from paper_2207_11571_gb300 import dg, nn

GAMMA, MACH, PR = 1.4, 0.1, 0.71
CS, PRT = 0.1, 0.9
RK_A, RK_B = (0.0, -5.0 / 9.0, -153.0 / 128.0), (1.0 / 3.0, 15.0 / 16.0, 8.0 / 15.0)


def _rk3(name, K, P, Re=1600.0, les=0, split=0, fp64=0, steps=1, io="none", width=0, hidden=0):
    c = {"kind": "rk3", "K": K, "P": P, "Re": Re, "les": les, "split": split, "fp64": fp64, "steps": steps, "io": io,
         "width": width, "hidden": hidden}
    return dict(c, name=name) if name else c


def _train(name, P, io, width, hidden, batch):
    c = {"kind": "train", "P": P, "io": io, "width": width, "hidden": hidden, "batch": batch}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the three benchmark meshes, one step per call, FP32 operator on the FP64 state
        _rk3("rk3_32c_P3", 32, 3),
        _rk3("rk3_16c_P6", 16, 6),
        _rk3("rk3_16c_P8", 16, 8),
        # the paper's own mesh at its moderate Reynolds number, several steps per call as
        # between two samples: small, bound by launches and latency
        _rk3("rk3_8c_P3_5steps", 8, 3, Re=200.0, steps=5),
        # a plain comparison run at an intermediate order with the Smagorinsky closure, on
        # a mesh of odd size (unaligned rows, ragged last blocks)
        _rk3("rk3_15c_P5_les", 15, 5, les=1),
        # the under-resolved high-order run of the paper's acceleration setting, kept stable
        # by the split-form volume term
        _rk3("rk3_8c_P8_split", 8, 8, split=1),
        # the FP64 operator, in which Algorithm 1's training window runs
        _rk3("rk3_16c_P3_fp64", 16, 3, les=1, fp64=1),
        # the corrected low-order run: network forcing in every stage (all five variables)
        _rk3("corrected_16c_P3_512x4", 16, 3, les=1, io="all", width=512, hidden=4),
        # a sweep over mesh, order and Reynolds number as one batch of twelve flows
        {"name": "batch_12", "kind": "batch",
         "members": "16/6/30 8/3/200 12/3/1600 8/6/1600 16/3/200 12/6/30 8/3/30 16/6/200 12/6/1600 8/6/200 16/3/1600 12/3/30"},
        # a sampling time of an evaluation run: P8 reference against the P3 run
        {"name": "sample_16c_P8_P3", "kind": "sample", "K": 16, "P_hi": 8, "P_lo": 3, "les": 1},
        # training the 512-wide network on all variables, batch 4096
        _train("train_320_512x4_b4096", 3, "all", 512, 4, 4096),
        # training the paper's 8-layer network on the momenta, small batch
        _train("train_192_256x7_b1024", 3, "momentum", 256, 7, 1024),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _mesh(rng, P, lo, hi):
    """Elements per direction for a node count spread over its logarithm in [lo, hi]."""
    return max(3, min(round(_log(rng, lo, hi) ** (1 / 3) / (P + 1)), int(hi ** (1 / 3) / (P + 1))))


def _flow(rng, K, P):
    """Reynolds number and closure; the high one only where mesh or closure carry it."""
    les = int(rng.random() < 0.4)
    return (rng.choice((30.0, 200.0, 1600.0)) if les or K * (P + 1) >= 96 else rng.choice((30.0, 200.0))), les


def draw(rng):
    u = rng.random()
    if u < 0.5:
        P = rng.randint(2, 8)
        fp64 = int(rng.random() < 0.2)
        K = _mesh(rng, P, 2e4, 4e5 if fp64 else 2.5e6)
        Re, les = _flow(rng, K, P)
        split = int(rng.random() < 0.2)
        return _rk3(None, K, P, Re, les, split, fp64, rng.choice((1, 1, 2, 5)) if K ** 3 * (P + 1) ** 3 < 2e5 else 1)
    if u < 0.65:
        P = rng.choice((2, 3, 3))
        K = _mesh(rng, P, 2e4, 4e5)
        return _rk3(None, K, P, 1600.0, 1, 0, 0, 1, rng.choice(("all", "momentum")), rng.choice((128, 256, 512)),
                    rng.randint(2, 7))
    if u < 0.75:
        left, members = 2.8e6, []
        for _ in range(rng.randint(2, 16)):
            P = rng.choice((2, 3, 3, 4, 5, 6, 6, 8))
            K = max(3, min(rng.randint(4, 16), int(max(left, 0) ** (1 / 3) / (P + 1))))
            left -= (K * (P + 1)) ** 3
            members.append("%d/%d/%d" % (K, P, rng.choice((30, 200, 1600))))
        return {"kind": "batch", "members": " ".join(members)}
    if u < 0.85:
        P_hi = rng.randint(4, 8)
        return {"kind": "sample", "K": _mesh(rng, P_hi, 2e4, 2.9e6), "P_hi": P_hi, "P_lo": rng.choice((2, 3)),
                "les": rng.randint(0, 1)}
    return _train(None, rng.choice((2, 3, 3)), rng.choice(("all", "momentum")), rng.choice((128, 256, 512)),
                  rng.randint(2, 7), int(_log(rng, 200, 4096)))


# ----------------------------------------------------------------------------- inputs

def _lobatto(P):
    """Gauss-Lobatto nodes, weights and derivative matrix of order P."""
    L = np.polynomial.legendre.Legendre.basis(P)
    x = np.concatenate([[-1.0], np.sort(L.deriv().roots().real), [1.0]])
    for _ in range(3):   # Newton on the inner nodes
        x[1:-1] -= L.deriv()(x[1:-1]) / L.deriv(2)(x[1:-1])
    w = 2.0 / (P * (P + 1) * L(x) ** 2)
    bary = np.array([1.0 / np.prod(x[i] - np.delete(x, i)) for i in range(P + 1)])
    D = np.zeros((P + 1, P + 1))
    for i in range(P + 1):
        for j in range(P + 1):
            if i != j:
                D[i, j] = bary[j] / bary[i] / (x[i] - x[j])
        D[i, i] = -D[i].sum()
    return x, w, D


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFF)
    return g


def _state(K, P, seed, salt):
    """Conserved state (5, K, K, K, n, n, n), axes (ez, ey, ex, k, j, i)."""
    x, _, _ = _lobatto(P)
    h, n = 2 * math.pi / K, P + 1
    c = torch.from_numpy(-math.pi + (np.arange(K)[:, None] + 0.5 * (x[None, :] + 1.0)) * h).cuda()
    X, Y, Z = c.view(1, 1, K, 1, 1, n), c.view(1, K, 1, 1, n, 1), c.view(K, 1, 1, n, 1, 1)
    rng = np.random.default_rng([int(seed), salt])
    one = torch.ones(K, K, K, n, n, n, dtype=torch.float64, device="cuda")
    u = torch.stack([torch.sin(X) * torch.cos(Y) * torch.cos(Z) * one, -torch.cos(X) * torch.sin(Y) * torch.cos(Z) * one,
                     0.0 * one])
    for _ in range(4):   # large-scale modes
        k = rng.integers(1, 4, 3)
        a, ph = 0.04 * rng.standard_normal(3), rng.uniform(0, 2 * math.pi, 3)
        mode = torch.sin(k[0] * X + ph[0]) * torch.sin(k[1] * Y + ph[1]) * torch.sin(k[2] * Z + ph[2])
        for v in range(3):
            u[v] += a[v] * mode
    p = 1.0 / (GAMMA * MACH * MACH) + (torch.cos(2 * X) + torch.cos(2 * Y)) * (torch.cos(2 * Z) + 2.0) / 16.0
    q = torch.stack([one, u[0], u[1], u[2], p / (GAMMA - 1.0) + 0.5 * (u * u).sum(0)])
    return q + 2e-4 * (torch.rand(q.shape, generator=_gen(seed, salt), dtype=torch.float64, device="cuda") - 0.5)


def _dt(K, P):
    """Acoustic CFL 0.4 for |v| + c up to 11.5 (the paper's steps on 8^3 elements are 0.37 to 0.6)."""
    return 0.4 * (2 * math.pi / K) / ((P + 1) ** 2 * 11.5)


def _io(io):
    return (1, 3) if io == "momentum" else (0, 5)


def _dims(case):
    feat = _io(case["io"])[1] * (case["P"] + 1) ** 3
    return [feat] + [case["width"]] * case["hidden"] + [feat]


def _draws(dims, seed):
    """U(-1, 1) draws of every dense layer, (out, in) FP32."""
    g = _gen(seed, 77)
    return [torch.rand((o, i), generator=g, device="cuda") * 2 - 1 for i, o in zip(dims[:-1], dims[1:])]


def _scalers(case, q):
    """FP32 feature scalers of a forcing network: inputs from the state's elements, a mild
    output amplitude."""
    f = _features(q, case["io"])
    feat = f.shape[1]
    return [f.mean(0).float().cpu().numpy(), (f.std(0, unbiased=False) + 1e-3).float().cpu().numpy(),
            np.zeros(feat, np.float32), np.full(feat, 0.01, np.float32)]


def _features(q, io):
    """Rows of one element: slot * n^3 + node."""
    first, nv = _io(io)
    K, np_ = q.shape[1], q.shape[4] ** 3
    return q[first:first + nv].reshape(nv, K ** 3, np_).transpose(0, 1).reshape(K ** 3, nv * np_)


def _pairs(case, seed):
    """Training rows (four mini-batches) and a shuffle of them."""
    g = _gen(seed, 5)
    rows, feat = 4 * case["batch"], _dims(case)[0]
    X = torch.randn((rows, feat), generator=g, device="cuda") * 0.5 + 0.1
    Y = torch.randn((rows, feat), generator=g, device="cuda") * 0.05
    return X, Y, torch.randperm(rows, generator=g, device="cuda")


class _Handle:
    """A library handle released with the state that holds it."""

    def __init__(self, h, free):
        self.h, self.free = h, free

    def __del__(self):
        self.free(self.h)


def _ctx(K, P, Re, les, fp64=0, split=0):
    return _Handle(dg.dg_create(K, P, Re, MACH, PR, les, precision=dg.DG_PREC_FP64 if fp64 else dg.DG_PREC_FP32,
                                volume_flux=split), dg.dg_destroy)


def _net(case, seed, max_batch):
    dims, (first, nv) = _dims(case), _io(case["io"])
    return _Handle(nn.nn_create(dims[0], dims[-1], case["width"], case["hidden"], first, nv, max_batch,
                                [w.cpu().numpy() for w in _draws(dims, seed)]), nn.nn_destroy)


def _members(case):
    return [(int(K), int(P), float(Re)) for K, P, Re in (m.split("/") for m in case["members"].split())]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rk3":
        q = _state(case["K"], case["P"], seed, 0)
        s = {"kind": kind, "ctx": _ctx(case["K"], case["P"], case["Re"], case["les"], case["fp64"], case["split"]),
             "net": None, "dt": _dt(case["K"], case["P"]), "steps": case["steps"]}
        if case["io"] != "none":
            s["net"] = _net(case, seed, 4096)
            nn.nn_set_scalers(s["net"].h, *_scalers(case, q))
        s["q"] = q.reshape(-1)
        return s
    if kind == "batch":
        ms = _members(case)
        return {"kind": kind, "dt": [_dt(K, P) for K, P, _ in ms],
                "q": [_state(K, P, seed, i).reshape(-1) for i, (K, P, _) in enumerate(ms)],
                "batch": _Handle(dg.dg_create_batch([(K, P, Re, MACH, PR, 0) for K, P, Re in ms],
                                                    precision=dg.DG_PREC_FP32), dg.dg_batch_destroy)}
    if kind == "sample":
        K, P_hi, P_lo = case["K"], case["P_hi"], case["P_lo"]
        q_lo = _state(K, P_lo, seed, 1).reshape(-1)
        return {"kind": kind, "hi": _ctx(K, P_hi, 1600.0, case["les"]), "lo": _ctx(K, P_lo, 1600.0, case["les"]),
                "q_hi": _state(K, P_hi, seed, 0).reshape(-1), "q_lo": q_lo, "qbar": torch.empty_like(q_lo)}
    X, Y, perm = _pairs(case, seed)
    net = _net(case, seed, case["batch"])
    nn.nn_compute_scalers(net.h, X, Y)
    grads = [g for l in range(case["hidden"] + 1) for g in nn.nn_grad_buffers(net.h, l)]
    for g in grads:
        g.owner = net   # views of the network's memory: they keep it
    return {"kind": kind, "net": net, "X": X, "Y": Y, "perm": perm, "batch": case["batch"], "at": 0, "grads": grads}


def run(state):
    kind = state["kind"]
    if kind == "rk3":
        dg.dg_rk3_step(state["ctx"].h, state["q"], state["dt"], state["steps"],
                       forcing=state["net"].h if state["net"] else None)
        return state["q"]
    if kind == "batch":
        dg.dg_batch_rk3_step(state["batch"].h, state["q"], state["dt"])
        return state["q"]
    if kind == "sample":
        dg.dg_project(state["hi"].h, state["lo"].h, state["q_hi"], state["qbar"])
        d_hi = dg.dg_diagnostics(state["hi"].h, state["q_hi"])
        d_lo = dg.dg_diagnostics(state["lo"].h, state["q_lo"], q_ref=state["qbar"])
        return {"qbar": state["qbar"], "hi": d_hi, "lo": d_lo}
    at, b = state["at"], state["batch"]
    nn.nn_train_step(state["net"].h, state["X"], state["Y"], state["perm"][at:at + b], want_loss=False)
    state["at"] = (at + b) % state["perm"].numel()
    return state["grads"]


def work(case):
    kind = case["kind"]

    def rk3(K, P, steps=1):
        N = (K * (P + 1)) ** 3
        return 80.0 * N, 3.0 * steps * (78 * (P + 1) + 300) * N

    def layers(dims, rows):
        return 2.0 * rows * sum(i * o for i, o in zip(dims[:-1], dims[1:])), sum(i * o + o for i, o in zip(dims[:-1], dims[1:]))

    if kind == "rk3":
        b, f = rk3(case["K"], case["P"], case["steps"])
        if case["io"] != "none":
            gf, params = layers(_dims(case), case["K"] ** 3)
            b, f = b + 2.0 * params, f + 3 * case["steps"] * gf
        return {"bytes": b, "flops": f}
    if kind == "batch":
        per = [rk3(K, P) for K, P, _ in _members(case)]
        return {"bytes": sum(b for b, _ in per), "flops": sum(f for _, f in per)}
    if kind == "sample":
        K, nh, nl = case["K"], case["P_hi"] + 1, case["P_lo"] + 1
        return {"bytes": 40.0 * K ** 3 * (nh ** 3 + 2 * nl ** 3),
                "flops": K ** 3 * (10.0 * nl * nh * (nh * nh + nl * nh + nl * nl)
                                   + sum((78 * n + 350) * n ** 3 for n in (nh, nl)))}
    gf, params = layers(_dims(case), case["batch"])
    # rows of X and Y; weights, moments read and written, gradients written
    return {"bytes": 8.0 * case["batch"] * _dims(case)[0] + 28.0 * params, "flops": 3 * gf}


# ----------------------------------------------------------------------------- 64 bits

class _Method:
    """The semi-discrete operator and RK3 in plain 64-bit torch on (5, K, K, K, n, n, n)."""

    def __init__(self, K, P, Re, les=0, split=0, forcing=None):
        _, w, D = _lobatto(P)
        self.K, self.n, self.w0, self.w = K, P + 1, float(w[0]), torch.from_numpy(w).cuda()
        self.D = torch.from_numpy(D).cuda()
        self.s = K / math.pi   # 2 / h
        self.mu, self.les, self.split, self.forcing = 1.0 / Re, les, split, forcing
        self.csd2 = (CS * 2 * math.pi / K / (P + 1)) ** 2

    def deriv(self, f, d):
        return torch.movedim(torch.movedim(f, -1 - d, -1) @ self.D.T, -1, -1 - d)

    def faces(self, f, d):
        """(own value at the right face, the right neighbour's at its left face)."""
        ax = f.dim() - 1 - d
        return f.select(ax, self.n - 1), torch.roll(f.select(ax, 0), -1, ax - 3)

    def prims(self, q):
        v = q[1:4] / q[0]
        return v, (GAMMA - 1) * (q[4] - 0.5 * (q[1:4] * v).sum(0))

    def euler(self, q, v, p, d):
        f = q * v[d]
        f[1 + d] += p
        f[4] += v[d] * p
        return f

    def roe(self, l, r, d):
        (vl, pl), (vr, pr) = self.prims(l), self.prims(r)
        a, b = torch.sqrt(l[0]), torch.sqrt(r[0])
        u = (a * vl + b * vr) / (a + b)
        H = (a * (l[4] + pl) / l[0] + b * (r[4] + pr) / r[0]) / (a + b)
        ke = 0.5 * (u * u).sum(0)
        c2 = (GAMMA - 1) * (H - ke)
        c, rho, du, dp, dr = torch.sqrt(c2), a * b, vr - vl, pr - pl, r[0] - l[0]
        w1 = (u[d] - c).abs() * (dp - rho * c * du[d]) / (2 * c2)
        w2 = u[d].abs()
        w5 = (u[d] + c).abs() * (dp + rho * c * du[d]) / (2 * c2)
        a2 = dr - dp / c2
        sh = rho * du
        sh[d] = 0
        m = (w1 + w5) * u + w2 * (a2 * u + sh)
        m[d] += (w5 - w1) * c
        E = w1 * (H - c * u[d]) + w2 * (a2 * ke + (u * sh).sum(0)) + w5 * (H + c * u[d])
        diss = torch.cat([(w1 + w2 * a2 + w5)[None], m, E[None]])
        return 0.5 * (self.euler(l, vl, pl, d) + self.euler(r, vr, pr, d) - diss)

    def kep(self, q, v, p, d):
        """2 sum_m D_im F#(i, m) with the two-point flux ({rho}{v_d}, m {v} + {p} e_d, m {H})."""
        ax, n = 5 - d, self.n
        w = torch.cat([q[:1], v, p[None], ((q[4] + p) / q[0])[None]])
        out = torch.zeros_like(q)
        for m in range(n):
            o = 0.5 * (w + w.narrow(ax + 1, m, 1))
            F = torch.empty_like(q)
            F[0] = o[0] * o[1 + d]
            F[1:4] = F[0] * o[1:4]
            F[1 + d] += o[4]
            F[4] = F[0] * o[5]
            shape = [1] * 7
            shape[ax + 1] = n
            out += 2 * self.D[:, m].reshape(shape) * F
        return out

    def rhs(self, q):
        n, lift = self.n, self.s / self.w0
        v, p = self.prims(q)
        U = torch.cat([v, (p / q[0])[None]])
        G = []
        for d in range(3):
            g, ax = self.s * self.deriv(U, d), 6 - d
            own, nb = self.faces(U, d)
            jump = 0.5 * lift * (nb - own)
            g.select(ax, n - 1).add_(jump)
            g.select(ax, 0).add_(torch.roll(jump, 1, ax - 3))
            G.append(g)
        mu = torch.full_like(p, self.mu)
        lam = mu * GAMMA / ((GAMMA - 1) * PR)
        if self.les:
            ss = sum((0.5 * (G[b][a] + G[a][b])) ** 2 for a in range(3) for b in range(3))
            mut = q[0] * self.csd2 * torch.sqrt(2 * ss)
            mu, lam = mu + mut, lam + mut * GAMMA / ((GAMMA - 1) * PRT)
        div = G[0][0] + G[1][1] + G[2][2]
        R = torch.zeros_like(q)
        for d in range(3):
            ax = 6 - d
            tau = torch.stack([mu * (G[d][a] + G[a][d]) for a in range(3)])
            tau[d] -= 2.0 / 3.0 * mu * div
            fv = torch.cat([torch.zeros_like(p)[None], tau, ((v * tau).sum(0) + lam * G[d][3])[None]])
            fa = self.euler(q, v, p, d)
            R -= self.s * ((self.kep(q, v, p, d) if self.split else self.deriv(fa, d)) - self.deriv(fv, d))
            (ql, qr), (vl, vr) = self.faces(q, d), self.faces(fv, d)
            star = self.roe(ql, qr, d) - 0.5 * (vl + vr)
            own = fa - fv
            R.select(ax, n - 1).sub_(lift * (star - own.select(ax, n - 1)))
            R.select(ax, 0).add_(lift * (torch.roll(star, 1, ax - 3) - own.select(ax, 0)))
        if self.forcing is not None:
            R += self.forcing(q)
        return R

    def steps(self, q, dt, count=1):
        g = torch.zeros_like(q)
        for _ in range(count):
            for a, b in zip(RK_A, RK_B):
                g = a * g + dt * self.rhs(q)
                q = q + b * g
        return q

    def diagnostics(self, q, ref=None):
        R = self.rhs(q)
        w = self.w
        W = (w.view(-1, 1, 1) * w.view(1, -1, 1) * w.view(1, 1, -1)) / self.s ** 3
        v, p = self.prims(q)
        v2, vol = (v * v).sum(0), (2 * math.pi) ** 3
        out = {"mass": W * q[0], "momentum": [W * q[1 + i] for i in range(3)], "energy": W * q[4],
               "ke": W * 0.5 * q[0] * v2 / vol, "dke_dt": W * ((v * R[1:4]).sum(0) - 0.5 * v2 * R[0]) / vol}
        out = {k: [float(x.sum()) for x in f] if isinstance(f, list) else float(f.sum()) for k, f in out.items()}
        out["e_inf"] = [float((q[1 + i] - ref[1 + i]).abs().max()) if ref is not None else 0.0 for i in range(3)]
        out["max_wave"] = float((torch.sqrt(v2) + torch.sqrt(GAMMA * p / q[0])).max())
        out["nonfinite"] = 0
        return out


def _weights(dims, seed):
    return [(w.cpu().double().numpy() * math.sqrt(6.0 / w.shape[1])).astype(np.float32) for w in _draws(dims, seed)]


def _filter(q, P_lo):
    """L2 projection of each element's polynomial to degree P_lo, at its own nodes."""
    P_hi = q.shape[-1] - 1
    x, w, _ = _lobatto(P_hi)
    xl = _lobatto(P_lo)[0]
    V = np.polynomial.legendre.legvander(x, P_hi)
    T = torch.from_numpy(np.polynomial.legendre.legvander(xl, P_lo) @ np.linalg.inv(V)[:P_lo + 1]).cuda()
    for d in range(3):
        q = torch.movedim(torch.movedim(q, -1 - d, -1) @ T.T, -1, -1 - d)
    return q.contiguous()


def exact(case, seed):
    kind = case["kind"]
    if kind == "rk3":
        K, P = case["K"], case["P"]
        q, net = _state(K, P, seed, 0), None
        if case["io"] != "none":
            first, nv = _io(case["io"])
            mi, si, mo, so = [torch.from_numpy(a).cuda().double() for a in _scalers(case, q)]
            Ws = [torch.from_numpy(w).cuda().double() for w in _weights(_dims(case), seed)]

            def net(z):
                a = (_features(z, case["io"]) - mi) / si
                for W in Ws[:-1]:
                    a = torch.relu(a @ W.T)
                a = (a @ Ws[-1].T) * so + mo
                s = torch.zeros_like(z)
                s[first:first + nv] = a.reshape(K ** 3, nv, -1).transpose(0, 1).reshape(nv, *z.shape[1:])
                return s
        m = _Method(K, P, case["Re"], case["les"], case["split"], net)
        return m.steps(q, _dt(K, P), case["steps"]).reshape(-1)
    if kind == "batch":
        return [_Method(K, P, Re).steps(_state(K, P, seed, i), _dt(K, P)).reshape(-1)
                for i, (K, P, Re) in enumerate(_members(case))]
    if kind == "sample":
        q_hi, q_lo = _state(case["K"], case["P_hi"], seed, 0), _state(case["K"], case["P_lo"], seed, 1)
        qbar = _filter(q_hi, case["P_lo"])
        return {"qbar": qbar.reshape(-1), "hi": _Method(case["K"], case["P_hi"], 1600.0, case["les"]).diagnostics(q_hi),
                "lo": _Method(case["K"], case["P_lo"], 1600.0, case["les"]).diagnostics(q_lo, qbar)}
    X, Y, perm = (t.double() if t.is_floating_point() else t for t in _pairs(case, seed))

    def scaled(A, rows):
        return (A[rows] - A.mean(0)) / A.std(0, unbiased=False)

    rows = perm[:case["batch"]]
    Ws = [torch.from_numpy(w).cuda().double() for w in _weights(_dims(case), seed)]
    acts = [scaled(X, rows)]
    for W in Ws[:-1]:
        acts.append(torch.relu(acts[-1] @ W.T))
    t = scaled(Y, rows)
    g = 2.0 * (acts[-1] @ Ws[-1].T - t) / t.numel()
    grads = []
    for l in range(len(Ws) - 1, -1, -1):
        grads = [g.T @ acts[l], g.sum(0)] + grads
        g = (g @ Ws[l]) * (acts[l] > 0)
    return grads
