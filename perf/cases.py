"""The work this framework is measured on, through its public entry points.

Every case is one call that a reconstruction program makes again and again:
the operator A_c and its adjoint, the data-consistency step of a DIP
iteration (eager and captured in a CUDA graph), the normal operator of a CG
iteration, the density compensation, a batch of several volumes, the TV
penalty with its gradient, and dictionary matching.  Sizes are those of the
workloads in `synth` and of the tests; `draw` covers the ranges between them,
odd and anisotropic matrices included.

A case is a dict of plain values.  `kind` names the call, `n1 n2 n3` the image,
`W`/`sigma` the gridding window, `K` the subspace channels, `C` the coils, `B`
the coil minibatch, `T` frames of `arms` arms of `arm_len` samples, `dcf`
whether the loss is density-compensated, and `shapes` whether the plan has the
default kernel shapes (a program that never ran the autotuner) or the ones the
autotuner picks at the benchmark's sizes.

`exact` is the same method in 64 bits, in plain torch: Kaiser-Bessel gridding
with the operator's own window placement, since a direct sum would measure the
gridding error (1e-3 at W = 4) and not the arithmetic.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2408_02367_gb300 import dm, graph, op, recon, synth

DEV = "cuda:0"

# The kernel shapes the autotuner picks at the benchmark's sizes.
TUNED = {"spread_bins": (4, 4, 4), "spread_chunk": 512, "fft_engine": 0, "fft_lines": 8, "fft_cols": 32,
         "fft_staged": 3, "interp_tiled": 1}

EPS_TV = 1e-6
DCF_ITERS = 10


# ----------------------------------------------------------------------------
# The cases
# ----------------------------------------------------------------------------

def _case(kind, n, W=4, sigma=1.25, K=5, C=8, B=2, T=480, arms=1, arm_len=1024, dcf=False, shapes="default", **more):
    return dict(kind=kind, n1=n[0], n2=n[1], n3=n[2], W=W, sigma=sigma, K=K, C=C, B=B, T=T, arms=arms,
                arm_len=arm_len, dcf=dcf, shapes=shapes, **more)


def _volumes(ws):
    """A batch of volumes as text: n1xn2xn3 C T arm_len B, separated by semicolons."""
    return ";".join("%dx%dx%d %d %d %d %d" % (*w[0], *w[1:]) for w in ws)


def listed():
    cases = {
        # the smallest DIP step of the test configurations: launches and latency count
        "dc_step_24_w6": _case("dc_step", (24, 24, 24), W=6, sigma=2.0, C=4, T=100, arm_len=512),
        # small accurate-mode forward: one k-space prediction of every coil
        "forward_32_w6": _case("forward", (32, 32, 32), W=6, sigma=2.0, C=4, B=4, T=100, arm_len=512),
        # the benchmark's DIP step as a plain program has it: default plan, eager autograd, with a DCF
        "dc_step_128": _case("dc_step", (128, 128, 128), dcf=True),
        # the benchmark's DIP step as a tuned program has it: captured in a CUDA graph
        "graph_step_128": _case("graph_step", (128, 128, 128), shapes="tuned"),
        # whole-brain DIP step, eight coils: the largest
        "dc_step_200x200x160": _case("dc_step", (200, 200, 160), C=32, B=8, T=1000, arms=2, shapes="tuned"),
        # a prescribed field of view: odd and unequal axes, an uneven minibatch
        "forward_111x90x77": _case("forward", (111, 90, 77), C=6, B=3, T=300, arm_len=1000),
        # the same in accurate mode, gradient direction, one coil
        "adjoint_75x64x90_w6": _case("adjoint", (75, 64, 90), W=6, sigma=2.0, C=4, B=1, T=250, arm_len=777),
        # one CG iteration's normal operator over all coils
        "normal_96": _case("normal", (96, 96, 96), B=4, T=400, dcf=True),
        # the Pipe-Menon density compensation of the 128^3 trajectory (one channel, no coils)
        "dcf_128": _case("dcf", (128, 128, 128), K=1, C=1, B=1),
        # one DIP step of several volumes at once (the four smaller ones of synth.MULTI_VOLUME)
        "batched_4_volumes": _case("batched", (0, 0, 0), shapes="tuned", volumes=_volumes(
            [(w.n, w.C, w.T, w.arm_len, w.batch) for w in synth.MULTI_VOLUME[:4]])),
        # the spatial penalty of a DIP step, value and gradient
        "tv_128": _case("tv", (128, 128, 128), C=1, B=1, T=16, arm_len=64),
        # Q-maps of a whole volume from a 9,438-atom dictionary
        "match_128": _case("match", (128, 128, 128), C=1, B=1, T=480, n_t1=128, n_t2=96),
    }
    return [dict(c, name=k) for k, c in cases.items()]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_image(rng, lo, hi):
    base = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return tuple(max(lo, int(round(base * rng.uniform(0.65, 1.0)))) for _ in range(3))


def draw(rng):
    kind = rng.choice(["forward", "forward", "adjoint", "adjoint", "dc_step", "dc_step", "dc_step", "graph_step",
                       "graph_step", "normal", "dcf", "batched", "tv", "match"])
    most = 0.8 * _cost(next(c for c in listed() if c["name"] == "dc_step_200x200x160"))
    while True:
        shapes = rng.choice(["default", "tuned"])
        W, sigma = rng.choice([(4, 1.25), (4, 1.25), (4, 1.25), (6, 2.0)])
        n = _draw_image(rng, 16, 200 if W == 4 else 100)
        K = rng.choice([5, 5, 5, rng.randint(1, 8)])
        B = rng.choice([1, 2, 3, 4, 8])
        T = _log_int(rng, 40, 1000)
        arm_len = rng.choice([256, 512, 1024, rng.randint(200, 1100)])
        arms = rng.choice([1, 1, 2])
        dcf = rng.random() < 0.3
        if kind == "dcf":
            c = _case(kind, n, W, sigma, K=1, C=1, B=1, T=T, arms=arms, arm_len=arm_len)
        elif kind == "tv":
            c = _case(kind, n, K=K, C=1, B=1, T=16, arm_len=64)
        elif kind == "match":
            c = _case(kind, _draw_image(rng, 16, 128), K=K, C=1, B=1, T=rng.randint(100, 480),
                      n_t1=rng.randint(24, 128), n_t2=rng.randint(24, 96))
        elif kind == "batched":
            vols = []
            for _ in range(rng.randint(2, 4)):
                Cv = rng.choice([4, 8, 16])
                vols.append((_draw_image(rng, 24, 140), Cv, _log_int(rng, 100, 600), 1024, max(1, Cv // 4)))
            c = _case(kind, (0, 0, 0), shapes=shapes, volumes=_volumes(vols))
        else:
            c = _case(kind, n, W, sigma, K=K, C=max(B, 4) if kind != "normal" else 2 * B, B=B, T=T, arms=arms,
                      arm_len=arm_len, dcf=dcf and kind != "graph_step", shapes=shapes)
        if _cost(c) <= most:
            return c


# ----------------------------------------------------------------------------
# Sizes and work
# ----------------------------------------------------------------------------

def _grid_len(n, sigma, W):
    m = max(math.ceil(sigma * n), 2 * W)
    while True:
        r = m
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if m % 2 == 0 and r == 1:
            return m
        m += 1


def _items(case):
    """The operators of a case: one, or those of a batch."""
    if case["kind"] != "batched":
        return [case]
    out = []
    for v in case["volumes"].split(";"):
        n, C, T, arm_len, B = v.split()
        out.append(_case("dc_step", [int(a) for a in n.split("x")], K=case["K"], C=int(C), B=int(B), T=int(T),
                         arm_len=int(arm_len), shapes=case["shapes"]))
    return out


def _sizes(c):
    n = (c["n1"], c["n2"], c["n3"])
    M = tuple(_grid_len(a, c["sigma"], c["W"]) for a in n)
    return n, M, int(np.prod(n)), int(np.prod(M)), c["T"] * c["arms"] * c["arm_len"]


def _one_way(c, coils):
    """Bytes and operations of the operator (or its adjoint) on `coils` coils: the image, the coil maps, the
    trajectory and the samples once; the FFTs of the gridding method and its window sums."""
    _, _, nvox, G, J = _sizes(c)
    byts = 8.0 * (c["K"] * nvox + coils * nvox + coils * J) + 16.0 * J + 8.0 * c["T"] * c["K"]
    flops = coils * c["K"] * (5.0 * G * math.log2(G) + 4.0 * J * c["W"] ** 3)
    return byts, flops


def work(case):
    kind = case["kind"]
    if kind == "tv":
        nvox = _sizes(case)[2]
        return {"bytes": 16.0 * case["K"] * nvox, "flops": 40.0 * case["K"] * nvox}
    if kind == "match":
        nvox = _sizes(case)[2]
        P = len(_dictionary(case["T"], case["K"], case["n_t1"], case["n_t2"])[0])
        return {"bytes": 8.0 * case["K"] * (nvox + P) + 20.0 * nvox, "flops": 8.0 * case["K"] * nvox * P}
    if kind == "dcf":
        J = _sizes(case)[4]
        return {"bytes": 20.0 * J, "flops": DCF_ITERS * 2.0 * 4.0 * J * case["W"] ** 3}
    byts = flops = 0.0
    for c in _items(case):
        coils = c["C"] if kind == "normal" else c["B"]
        b, f = _one_way(c, coils)
        two = kind not in ("forward", "adjoint")
        byts += b + (8.0 * c["K"] * _sizes(c)[2] if two else 0.0)
        flops += f * (2 if two else 1)
    return {"bytes": byts, "flops": flops}


def _cost(case):
    """What a pass costs, roughly, for the comparison of two cases: its operations, an untuned plan's counted twice."""
    w = {"flops": 3e3 * _sizes(case)[2]} if case["kind"] == "match" else work(case)
    return w["flops"] * (2 if case["shapes"] == "default" else 1)


# ----------------------------------------------------------------------------
# Inputs (made on the GPU from the seed)
# ----------------------------------------------------------------------------

def _gen(seed, stream):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1000 + stream)


def _cgauss(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device=DEV)) / math.sqrt(2.0)


def _coords(n):
    return [(torch.arange(a, device=DEV, dtype=torch.float32) - a // 2) / (a / 2.0) for a in n]


def _phantom(n, K, seed):
    """A dozen soft-edged ellipsoids with complex amplitudes falling over the channels."""
    rng = np.random.default_rng([seed, 11])
    u = _coords(n)
    x = torch.zeros((K,) + tuple(n), dtype=torch.complex64, device=DEV)
    for _ in range(12):
        ctr, ax = rng.uniform(-0.6, 0.6, 3), rng.uniform(0.1, 0.45, 3)
        q = np.linalg.qr(rng.standard_normal((3, 3)))[0]
        amp = (rng.standard_normal(K) + 1j * rng.standard_normal(K)) / math.sqrt(2.0) / (np.arange(K) + 1.0)
        d = [u[0][:, None, None] - ctr[0], u[1][None, :, None] - ctr[1], u[2][None, None, :] - ctr[2]]
        r2 = sum(((float(q[0, j]) * d[0] + float(q[1, j]) * d[1] + float(q[2, j]) * d[2]) / float(ax[j])) ** 2
                 for j in range(3))
        soft = torch.sigmoid((1.0 - r2) * 10.0)
        x += torch.from_numpy(amp.astype(np.complex64)).to(DEV)[:, None, None, None] * soft
    return x


def _coil_maps(n, C, seed):
    """Gaussian-bump sensitivities around the volume, unit root-sum-of-squares."""
    turn = np.random.default_rng([seed, 12]).uniform(0.0, 2.0 * np.pi)
    u = _coords(n)
    S = torch.empty((C,) + tuple(n), dtype=torch.complex64, device=DEV)
    for c in range(C):
        z = 1.0 - 2.0 * (c + 0.5) / C
        a = np.pi * (3.0 - math.sqrt(5.0)) * c + turn
        r = math.sqrt(max(0.0, 1.0 - z * z))
        d = 1.2 * np.array([r * math.cos(a), r * math.sin(a), z])
        p = [torch.polar(torch.exp(-(v - float(d[i])) ** 2 / 2.88), 0.3 * float(d[i]) * v) for i, v in enumerate(u)]
        p[0] = p[0] * complex(math.cos(2 * math.pi * c / C), math.sin(2 * math.pi * c / C))
        S[c] = p[0][:, None, None] * p[1][None, :, None] * p[2][None, None, :]
    S /= torch.linalg.vector_norm(S, dim=0)
    return S


def _trajectory(T, arms, arm_len, seed):
    """Golden-angle spiral arms in 3D (as synth.spiral_trajectory has them), the whole set turned by the seed."""
    n = T * arms
    p1, p2 = synth.golden_means_3d()
    i = torch.arange(n, dtype=torch.float64, device=DEV)
    cz = 2.0 * torch.remainder(i * p1, 1.0) - 1.0
    az = 2.0 * math.pi * torch.remainder(i * p2, 1.0)
    sz = torch.sqrt(torch.clamp(1.0 - cz * cz, min=0.0))
    nrm = torch.stack([sz * torch.cos(az), sz * torch.sin(az), cz], 1)
    ref = torch.where(nrm[:, 2:].abs() < 0.9, torch.tensor([[0.0, 0.0, 1.0]], dtype=torch.float64, device=DEV),
                      torch.tensor([[1.0, 0.0, 0.0]], dtype=torch.float64, device=DEV))
    e1 = torch.linalg.cross(nrm, ref)
    e1 = e1 / torch.linalg.vector_norm(e1, dim=1, keepdim=True)
    e2 = torch.linalg.cross(nrm, e1)
    turn = np.linalg.qr(np.random.default_rng([seed, 13]).standard_normal((3, 3)))[0]
    turn = torch.from_numpy(turn).to(DEV)
    s = torch.arange(arm_len, dtype=torch.float64, device=DEV) / max(arm_len - 1, 1)
    ang = 2.0 * math.pi * (arm_len / 64.0) * s[None, :] + (math.pi * (3.0 - math.sqrt(5.0)) * i)[:, None]
    k = (math.pi * s)[None, :, None] * (torch.cos(ang)[..., None] * (e1 @ turn)[:, None, :]
                                        + torch.sin(ang)[..., None] * (e2 @ turn)[:, None, :])
    omega = k.reshape(-1, 3).clamp(-math.pi, math.pi).to(torch.float32).contiguous()
    return omega, np.arange(T + 1, dtype=np.int64) * (arms * arm_len)


def _kspace(omega, rows, nvox, seed):
    """Measured samples: random, with the magnitude of k-space data (large at the centre)."""
    r = torch.linalg.vector_norm(omega, dim=1) / math.pi
    env = 0.05 * nvox / (1.0 + (r / 0.04) ** 2) + 0.3 * math.sqrt(nvox)
    y = _cgauss((rows, omega.shape[0]), _gen(seed, 14))
    return y.mul_(env[None, :])


def _inputs(c, seed):
    n, _, nvox, _, J = _sizes(c)
    omega, off = _trajectory(c["T"], c["arms"], c["arm_len"], seed)
    ones = c["kind"] == "dcf"
    d = {"n": n, "omega": omega, "off": off, "J": J,
         "V": torch.from_numpy(synth.subspace_basis(c["T"], c["K"], seed=seed + 20)).to(DEV) if not ones else None,
         "S": _coil_maps(n, c["C"], seed) if not ones else None}
    if ones:
        return d
    coils = np.sort(np.random.default_rng([seed, 15]).choice(c["C"], size=c["B"], replace=False)).astype(np.int32)
    d["coils"] = torch.from_numpy(coils).to(DEV)
    d["x"] = _phantom(n, c["K"], seed)
    if c["kind"] != "forward":
        rows = c["B"] if c["kind"] == "adjoint" else c["C"]
        d["y"] = _kspace(omega, rows, nvox, seed)
    d["dcf"] = (torch.linalg.vector_norm(omega, dim=1) / math.pi).square_().add_(1e-3) if c["dcf"] else None
    return d


def _plan(c, d):
    return op.SubspaceNufft(d["omega"], d["off"], d["n"], c["W"], c["sigma"], d["V"], d["S"], max_batch=c["B"],
                            tuning=TUNED if c["shapes"] == "tuned" else None, borrow_maps=True)


@functools.lru_cache(maxsize=None)
def _dictionary(T, K, n_t1, n_t2):
    """The compressed dictionary (atoms [P][K]) and its (T1, T2) table, on the host."""
    f, params = synth.mrf_dictionary(T, n_t1, n_t2)
    f = f.astype(np.complex128)
    w, v = np.linalg.eigh(f.T @ f.conj())
    V = v[:, ::-1][:, :K].conj()
    return np.ascontiguousarray((f @ V.conj()).astype(np.complex64)), params


def prepare(case, seed):
    kind = case["kind"]
    if kind == "match":
        n, _, nvox, _, _ = _sizes(case)
        atoms, params = _dictionary(case["T"], case["K"], case["n_t1"], case["n_t2"])
        at = torch.from_numpy(atoms).to(DEV)
        g = _gen(seed, 16)
        p = torch.randint(at.shape[0], (nvox,), generator=g, device=DEV)
        mag = 0.5 + 1.5 * torch.rand(nvox, generator=g, device=DEV)
        pd = torch.polar(mag, 2 * math.pi * torch.rand(nvox, generator=g, device=DEV))
        x = (pd[:, None] * at[p]).T
        noise = 0.01 * torch.linalg.vector_norm(x, dim=0).mean() / math.sqrt(case["K"])
        x = (x + noise * _cgauss(x.shape, g)).reshape((case["K"],) + n).contiguous()
        return {"kind": kind, "x": x,
                "m": dm.DictionaryMatcher(at, max_vox=nvox, params=torch.from_numpy(params).to(DEV))}
    if kind == "dcf":
        d = _inputs(case, seed)
        return {"kind": kind, "A": recon.dcf_operator(d["omega"].cpu().numpy(), d["n"], case["W"], case["sigma"],
                                                      device=DEV)}
    items = []
    for i, c in enumerate(_items(case)):
        d = _inputs(c, seed + 100 * i)
        d["A"] = _plan(c, d)
        items.append(d)
    d = items[0]
    if kind in ("dc_step", "tv"):
        d["x"].requires_grad_(True)
    state = {"kind": kind, "items": items}
    if kind == "graph_step":
        state["graph"] = graph.DipStepGraph(d["A"], d["y"], d["x"], B=case["B"])
    return state


# ----------------------------------------------------------------------------
# One pass
# ----------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "match":
        return state["m"].match(state["x"], qmap=True)
    if kind == "dcf":
        return recon.dcf_pipe_menon(state["A"], iters=DCF_ITERS)
    d = state["items"][0]
    A = d["A"]
    if kind == "forward":
        return A.forward(d["x"], d["coils"])
    if kind == "adjoint":
        return A.adjoint(d["y"], d["coils"])
    if kind == "normal":
        return recon.normal_apply(A, d["x"], d["dcf"])
    if kind == "graph_step":
        loss, grad = state["graph"].step(d["coils"], x=d["x"])
        return loss, grad
    if kind == "batched":
        ys = op.forward_batched([(e["A"], e["x"], e["coils"], None) for e in state["items"]])
        res = [e["A"].residual_loss(y, e["y"], e["coils"]) for e, y in zip(state["items"], ys)]
        grads = op.adjoint_batched([(e["A"], r2, e["coils"], None, False) for e, (r2, _) in zip(state["items"], res)])
        return [loss for _, loss in res], grads
    x = d["x"]
    x.grad = None
    loss = op.tv_loss(A, x, 1e-3, EPS_TV) if kind == "tv" else op.dc_loss(A, x, d["coils"], d["y"], dcf=d["dcf"])
    loss.backward()
    return loss.detach(), x.grad


# ----------------------------------------------------------------------------
# The same in 64 bits
# ----------------------------------------------------------------------------

class _Gridding:
    """Kaiser-Bessel gridding in float64: the operator of one case on its trajectory."""

    def __init__(self, c, omega):
        self.n, self.M, _, self.G, self.J = _sizes(c)
        self.W, self.sigma = c["W"], c["sigma"]
        beta = math.pi * math.sqrt((self.W / self.sigma) ** 2 * (self.sigma - 0.5) ** 2 - 0.8)
        i0b = float(np.i0(beta))
        self.idx, self.wt, self.dinv = [], [], []
        for a in range(3):
            m = float(self.M[a])
            g = omega[:, a].double() * (m / (2.0 * math.pi))
            g = torch.where(g < 0, g + m, g)
            g = torch.where(g >= m, g - m, g).float()
            g = torch.where(g >= m, torch.zeros_like(g), g)
            m0 = torch.ceil(g - 0.5 * self.W).double()     # the window's start, decided in float32
            taps = m0[:, None] + torch.arange(self.W, device=DEV, dtype=torch.float64)
            q = 2.0 * (g.double()[:, None] - taps) / self.W
            self.wt.append(torch.special.i0(beta * torch.sqrt(torch.clamp(1.0 - q * q, min=0.0))) / i0b)
            self.idx.append(torch.remainder(taps, m).long())
            xi = (torch.arange(self.n[a], dtype=torch.float64) - self.n[a] // 2) / m
            z2 = beta ** 2 - (math.pi * self.W * xi) ** 2
            z = torch.sqrt(z2.abs())
            ft = torch.where(z2 > 0, torch.sinh(z), torch.sin(z)) / z
            self.dinv.append((i0b / (self.W * ft)).to(DEV))

    def _taps(self):
        M2, M3 = self.M[1], self.M[2]
        for a in range(self.W):
            for b in range(self.W):
                row = (self.idx[0][:, a] * M2 + self.idx[1][:, b]) * M3
                w = self.wt[0][:, a] * self.wt[1][:, b]
                for c in range(self.W):
                    yield row + self.idx[2][:, c], w * self.wt[2][:, c]

    def interp(self, grid):
        """grid [K][G] complex128 -> [K][J]."""
        out = torch.zeros((grid.shape[0], self.J), dtype=torch.complex128, device=DEV)
        for at, w in self._taps():
            out += grid[:, at] * w
        return out

    def spread(self, z):
        """z [K][J] -> [K][G]."""
        grid = torch.zeros((z.shape[0], self.G, 2), dtype=torch.float64, device=DEV)
        zr = torch.view_as_real(z)
        for at, w in self._taps():
            grid.index_add_(1, at, zr * w[:, None])
        return torch.view_as_complex(grid)

    def _window(self):
        """Where the image sits in the grid, and 1 / psi_hat."""
        at = [torch.remainder(torch.arange(n, device=DEV) - n // 2, M) for n, M in zip(self.n, self.M)]
        d = self.dinv
        return (slice(None), at[0][:, None, None], at[1][None, :, None], at[2][None, None, :]), \
            d[0][:, None, None] * d[1][None, :, None] * d[2][None, None, :]

    def forward(self, x, S, V):
        at, dinv = self._window()
        grid = torch.zeros((x.shape[0],) + self.M, dtype=torch.complex128, device=DEV)
        grid[at] = x * (S * dinv)
        grid = torch.fft.fftn(grid, dim=(1, 2, 3)).reshape(x.shape[0], -1)
        return (self.interp(grid) * V.T).sum(0)

    def adjoint(self, y, S, V):
        at, dinv = self._window()
        grid = self.spread(V.conj().T * y).reshape((V.shape[1],) + self.M)
        grid = torch.fft.ifftn(grid, dim=(1, 2, 3), norm="forward")
        return grid[at] * (S.conj() * dinv)


def _exact_operator(c, d, kind):
    A = _Gridding(c, d["omega"])
    per = c["arms"] * c["arm_len"]
    V = d["V"].to(torch.complex128).repeat_interleave(per, 0)
    maps = lambda k: d["S"][k].to(torch.complex128)  # noqa: E731
    coils = [int(k) for k in d["coils"].cpu()]
    x = d["x"].to(torch.complex128)
    w = d["dcf"].double() if d["dcf"] is not None else 1.0
    if kind == "forward":
        return torch.stack([A.forward(x, maps(k), V) for k in coils])
    out = torch.zeros_like(x)
    if kind == "adjoint":
        for b, k in enumerate(coils):
            out += A.adjoint(d["y"][b].to(torch.complex128), maps(k), V)
        return out
    if kind == "normal":
        for k in range(c["C"]):
            out += A.adjoint(A.forward(x, maps(k), V) * w, maps(k), V)
        return out
    loss = 0.0
    for k in coils:
        r = A.forward(x, maps(k), V) - d["y"][k].to(torch.complex128)
        loss = loss + (w * r.abs() ** 2).sum()
        out += A.adjoint(2.0 * w * r, maps(k), V)
    return loss, out


def exact(case, seed):
    kind = case["kind"]
    if kind == "match":
        return None     # the matched atom is a choice among near ties
    if kind == "dcf":
        A = _Gridding(case, _inputs(case, seed)["omega"])
        w = torch.ones((1, A.J), dtype=torch.complex128, device=DEV)
        for _ in range(DCF_ITERS):
            w = (w.real / A.interp(A.spread(w)).real).to(torch.complex128)
        return w.real[0].contiguous()
    if kind == "tv":
        x = _phantom(_sizes(case)[0], case["K"], seed).to(torch.complex128).requires_grad_(True)
        s = EPS_TV ** 2
        for a in (1, 2, 3):
            d = torch.diff(x, dim=a, append=x.narrow(a, x.shape[a] - 1, 1))
            s = s + d.real ** 2 + d.imag ** 2
        loss = 1e-3 * torch.sqrt(s).sum()
        loss.backward()
        return loss.detach(), x.grad
    got = [_exact_operator(c, _inputs(c, seed + 100 * i), "dc_step" if kind in ("graph_step", "batched") else kind)
           for i, c in enumerate(_items(case))]
    return [[g[0] for g in got], [g[1] for g in got]] if kind == "batched" else got[0]
