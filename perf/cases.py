"""The work a user of the solver has it do, as cases that can be timed and compared.

A case is a dict of plain values; prepare() builds its inputs on the GPU from a seed
(initial data of the runs this repository is tested and benchmarked on, carried a few
time steps forward by the spectral solver below so that the history and the velocity are
those of a running simulation), run() is one pass through the public entry points, and
exact() gives the same results in plain 64-bit torch.
"""
import ctypes
import math
import random

import numpy as np
import torch

from paper_1208_2643_gb300 import guess, inputs, mpfc

DEV = "cuda"
NOISE = dict(init="noise", mean=0.07, h=0.5, dt=0.01, epsilon=0.025, beta=0.9, M=1.0)
CRYSTAL = dict(init="crystal", mean=-0.285, h=math.pi / 4, dt=0.05, epsilon=0.25, beta=0.9, M=1.0)


def _step(name, m, n, scheme, steps, base, **kw):
    c = dict(kind="step", m=m, n=n, scheme=scheme, steps=steps, precision="fp64", inner=0, bc="periodic", model="mpfc",
             guess="extrap", pinned=False, burn=3, **base)
    c.update(kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest grid of the repository's workloads: four steps of a short-box run, where launches,
        # latency and the call itself count
        _step("fp64_64", 64, 64, 1, 4, NOISE),
        # the benchmark's headline grid, first-order scheme, two steps of a run
        _step("fp64_1024", 1024, 1024, 1, 2, NOISE),
        # second-order scheme on growing crystallites, the 512^2 production run of Sec. 4
        _step("fp64_s2_512", 512, 512, 2, 4, CRYSTAL),
        # a strained crystal held by pinned strips (Sec. 4.6), a grid that is not a square or a power of two
        _step("fp64_pinned_512x384", 512, 384, 2, 2,
              dict(init="slab", mean=0.57, h=4 * math.pi / (16 * math.sqrt(3.0)), dt=0.00513, epsilon=0.6, beta=0.2, M=225.0),
              pinned=True),
        # the polycrystal run of Sec. 4.5: mixed boundaries and a time step of 1, many V-cycles per step
        _step("fp64_neumann_2048", 2048, 2048, 2, 1,
              dict(CRYSTAL, mean=0.285, h=804.0 / 2048.0, dt=1.0), bc="neumann", burn=1),
        # the largest everyday grid: one step of a 4096^2 run
        _step("fp64_4096", 4096, 4096, 1, 1, NOISE, burn=2),
        # the mixed-precision form on the headline grid and on the large one with the larger time step
        _step("mixed_1024", 1024, 1024, 1, 2, NOISE, precision="fp32_inner", inner=2),
        _step("mixed_2048", 2048, 2048, 1, 2, dict(NOISE, dt=0.02), precision="fp32_inner", inner=3),
        # steps whose guess a trained network corrects
        _step("learned_1024", 1024, 1024, 1, 2, NOISE, guess="learned"),
        # a parameter study: instances of uneven size advanced together
        dict(name="ensemble_16", kind="batch", count=16, largest=1024, scheme=1, steps=1, pick=4),
        # energies and mass of a state, as a run logs them every few steps
        dict(_step("energy_1024", 1024, 1024, 2, 0, CRYSTAL, burn=1), kind="energy"),
        # one optimiser step of the guess network on a batch of 256^2 fields
        dict(name="train_8x256", kind="train", B=8, H=256, W=256),
    ]


def _sizes(rng, cells):
    """A grid of about `cells` cells that the hierarchy takes: both sides (even) * 2^k, at most 64 cells coarsest."""
    shapes = [(4, 4), (6, 6), (8, 8), (4, 6), (6, 4), (6, 8), (8, 6), (4, 8), (8, 4), (6, 10), (10, 6), (4, 12), (4, 14), (14, 4), (4, 16)]
    a, b = rng.choice(shapes)
    k = max(2, round(0.5 * math.log2(cells / (a * b))))
    return a << k, b << k


def draw(rng):
    u = rng.random()
    if u < 0.12:
        return dict(kind="batch", count=rng.randint(3, 16), largest=rng.choice([128, 256, 512]), scheme=rng.choice([1, 2]),
                    steps=rng.randint(1, 2), pick=rng.randint(1, 1 << 20))
    if u < 0.2:
        return dict(kind="train", B=rng.randint(1, 8), H=8 * rng.randint(4, 32), W=rng.choice([40, 64, 72, 128, 200, 256]))
    m, n = _sizes(rng, 2.0 ** rng.uniform(12, 22.5))
    scheme = rng.choice([1, 2])
    base = dict(NOISE, mean=rng.uniform(0.05, 0.1), dt=10 ** rng.uniform(-2.3, -1.3), epsilon=rng.uniform(0.02, 0.1),
                beta=rng.uniform(0.5, 1.5), h=rng.choice([0.4, 0.5, 0.6])) if rng.random() < 0.5 else dict(
                    CRYSTAL, mean=rng.choice([-0.285, 0.285]), dt=10 ** rng.uniform(-1.7, 0.0), h=rng.uniform(0.4, 0.8))
    if u < 0.28:
        return dict(_step("", m, n, 2, 0, base, burn=1), kind="energy")
    c = _step("", m, n, scheme, rng.randint(1, 3), base)
    v = rng.random()
    if v < 0.3:
        c.update(precision="fp32_inner", inner=rng.randint(2, 4))
    elif v < 0.4:
        c.update(guess="prev")
    if rng.random() < 0.25:
        c.update(bc="neumann")
    if rng.random() < 0.15:
        c.update(model="pfc")
    elif scheme == 2 and rng.random() < 0.25:
        c.update(pinned=True)
    return c


# ------------------------------------------------------------------------- inputs
def _noise(m, n, mean, amp, seed):
    return inputs.noise_field_torch(m, n, mean, amp, seed, device=DEV)


def _pattern(c, x, y, shift=0.0):
    """One-mode hexagonal density about |mean| (Sec. 4.6, (4.4)-(4.5)), without its mean."""
    A = inputs.single_mode_amplitude(abs(c["mean"]), c["epsilon"])
    q = math.sqrt(3.0) / 2.0
    return A * (torch.cos(q * (x - shift)) * torch.cos(q * y / math.sqrt(3.0)) - 0.5 * torch.cos(2 * q * y / math.sqrt(3.0)))


def _axes(c):
    x = (torch.arange(c["m"], dtype=torch.float64, device=DEV) + 0.5) * c["h"]
    y = (torch.arange(c["n"], dtype=torch.float64, device=DEV) + 0.5) * c["h"]
    return x[None, :], y[:, None]


def _initial(c, seed):
    """phi of the run's start, from the seed."""
    m, n, h, mean = c["m"], c["n"], c["h"], c["mean"]
    if c["init"] == "noise":
        return _noise(m, n, mean, 0.05, seed)
    x, y = _axes(c)
    rng = random.Random(seed)
    dev = torch.zeros(n, m, dtype=torch.float64, device=DEV)
    if c["init"] == "slab":
        j = torch.arange(n, device=DEV)[:, None]
        dev = torch.where((j >= n // 5) & (j < n - n // 5), _pattern(c, x, y, rng.uniform(0, 2)), dev)
    else:
        for _ in range(3):   # rotated crystallites in a uniform liquid
            cx, cy, th = rng.random() * m * h, rng.random() * n * h, rng.random() * math.pi / 3
            dx = torch.remainder(x - cx + 0.5 * m * h, m * h) - 0.5 * m * h
            dy = torch.remainder(y - cy + 0.5 * n * h, n * h) - 0.5 * n * h
            pat = _pattern(c, math.cos(th) * dx + math.sin(th) * dy, math.cos(th) * dy - math.sin(th) * dx)
            dev = torch.where(dx * dx + dy * dy <= (0.2 * min(m, n) * h) ** 2, pat, dev)
    return (abs(mean) + dev) * (1 if mean >= 0 else -1) + _noise(m, n, 0.0, 1e-3, seed + 17)


def _pins(c):
    """Weight 2 in strips at the slab's top and bottom, target sheared by 4 % of 2 pi."""
    if not c["pinned"]:
        return None, None
    n, strip = c["n"], max(2, round(math.pi / c["h"]))
    x, y = _axes(c)
    W = torch.zeros(n, c["m"], dtype=torch.float64, device=DEV)
    lo, hi = n // 5, n - n // 5
    W[lo:lo + strip] = 2.0
    W[hi - strip:hi] = 2.0
    shift = torch.where(y > 0.5 * n * c["h"], 0.04 * 2 * math.pi, 0.0)
    return W, abs(c["mean"]) + _pattern(c, x, y, shift)


# ------------------------------------------------- the schemes of Sec. 3, spectral, 64 bits
class _Spectral:
    """phi^{k+1} of the convex-splitting schemes by a fixed-point iteration on the constant-coefficient
    part of phi = S1 + c L (S2 + g(phi) + (gam + W) phi + L (S3 + theta L phi)), L the five-point Laplacian."""

    def __init__(self, c, W=None, target=None):
        self.c, self.W, self.target = c, W, target
        m, n, h = c["m"], c["n"], c["h"]
        self.n, self.even = n, c.get("bc") == "neumann"
        rows = 2 * n if self.even else n
        f = lambda k: 4.0 / (h * h) * torch.sin(math.pi * torch.arange(k, dtype=torch.float64, device=DEV) / k) ** 2  # noqa: E731
        self.lam = -(f(rows)[:, None] + f(m)[None, : m // 2 + 1])

    def fwd(self, a):
        return torch.fft.rfft2(torch.cat([a, a.flip(0)]) if self.even else a)

    def inv(self, a):
        return torch.fft.irfft2(a, s=(2 * self.n if self.even else self.n, self.c["m"]))[: self.n]

    def lap(self, a):
        up = torch.cat([a[1:], a[-1:]]) if self.even else a.roll(-1, 0)
        down = torch.cat([a[:1], a[:-1]]) if self.even else a.roll(1, 0)
        return (up + down + a.roll(1, 1) + a.roll(-1, 1) - 4.0 * a) / self.c["h"] ** 2

    def step(self, pk, pm, psi):
        c, s = self.c, self.c["dt"]
        s2, pfc, alpha = c["scheme"] == 2, c["model"] == "pfc", 1.0 - c["epsilon"]
        damp = c["beta"] + (2.0 if s2 else 1.0) / s
        cc = s * c["M"] if pfc else s * c["M"] / damp
        S1 = pk if pfc else pk + ((2.0 if s2 else 1.0) / damp) * psi
        if s2:
            gam, theta, S3 = 0.5 * alpha, 0.5, 0.5 * self.lap(pk)
            S2 = 0.5 * alpha * pk + 2.0 * self.lap(1.5 * pk - 0.5 * pm)
            if self.W is not None:
                S2 = S2 + self.W * (pk - 2.0 * self.target)
        else:
            gam, theta, S2, S3 = alpha, 1.0, 2.0 * self.lap(pk), None

        def g(p):
            return 0.25 * (p * p + pk * pk) * (p + pk) if s2 else p * p * p

        q = float((0.25 * (6.0 * pk * pk) if s2 else 3.0 * pk * pk).mean())
        lam = self.lam
        den = 1.0 - cc * (gam + q) * lam - cc * theta * lam ** 3
        rhs = self.fwd(S1) + cc * lam * self.fwd(S2 if S3 is None else S2 + self.lap(S3))
        p = 2.0 * pk - pm
        for _ in range(80):
            rest = g(p) - q * p
            if s2 and self.W is not None:
                rest = rest + self.W * p
            new = self.inv((rhs + cc * lam * self.fwd(rest)) / den)
            d = float((new - p).abs().max())
            p = new
            if d < 2e-15:
                break
        if s2 and not pfc:
            v = (2.0 / s) * (p - pk) - psi
        else:
            v = (p - pk) / s
        return p, pk, v


def _state(c, seed):
    """(phi^k, phi^{k-1}, psi^k, W, target) a few steps into a run."""
    W, target = _pins(c)
    sp = _Spectral(c, W, target)
    phi = _initial(c, seed)
    st = (phi, phi, torch.zeros_like(phi))
    for _ in range(c["burn"]):
        st = sp.step(*st)
    return [a.contiguous() for a in st], W, target, sp


def _instances(c, seed):
    """The batch's instances: the ensemble workload's sizes and parameters, seeded noise."""
    pick = random.Random(c["pick"])
    sizes = [s for s in (128, 256, 512, 1024) if s <= c["largest"]]
    out = []
    for i in range(c["count"]):
        m = pick.choice(sizes)
        n = m if pick.random() < 0.75 else m // 2
        out.append(dict(kind="step", m=m, n=n, scheme=c["scheme"], h=0.5, dt=0.01, epsilon=pick.uniform(0.02, 0.1),
                        beta=pick.uniform(0.5, 1.5), M=1.0, mean=pick.uniform(0.05, 0.1), init="noise", model="mpfc",
                        bc="periodic", pinned=False, burn=1, seed=seed * 1000 + i))
    return out


def _params(c):
    return mpfc.default_params(
        m=c["m"], n=c["n"], h=c["h"], dt=c["dt"], M=c["M"], epsilon=c["epsilon"], beta=c["beta"],
        precision=mpfc.MPFC_FP32_INNER if c.get("precision") == "fp32_inner" else mpfc.MPFC_FP64, inner_cycles=c.get("inner", 0),
        guess={"prev": mpfc.MPFC_GUESS_PREV, "learned": mpfc.MPFC_GUESS_LEARNED}.get(c.get("guess"), mpfc.MPFC_GUESS_EXTRAP),
        bc=mpfc.MPFC_BC_NEUMANN_Y if c["bc"] == "neumann" else mpfc.MPFC_BC_PERIODIC, pinning=int(c["pinned"]),
        model=mpfc.MPFC_MODEL_PFC if c["model"] == "pfc" else mpfc.MPFC_MODEL_MPFC)


def _samples(c, seed):
    """Four successive fields of each sample of a training batch, phi^{k-2} .. phi^{k+1}."""
    B, H, W = c["B"], c["H"], c["W"]
    f = [torch.empty(B, H, W, dtype=torch.float64, device=DEV) for _ in range(4)]
    rng = random.Random(seed)
    for b in range(B):
        one = dict(NOISE, m=W, n=H, scheme=1, model="mpfc", bc="periodic", epsilon=rng.uniform(0.02, 0.1),
                   mean=rng.uniform(0.05, 0.1))
        sp = _Spectral(one)
        st = (_initial(one, seed * 100 + b),) * 2 + (torch.zeros(H, W, dtype=torch.float64, device=DEV),)
        for k in range(4):
            st = sp.step(*st)
            f[k][b] = st[0]
    return f


def _blob():
    """A model early in training: the initial weights, an output layer that has begun to move, the
    packaged model's normalisation scales."""
    blob = guess.init_params(0)
    blob[:4] = guess.load()[:4]
    w = guess.layer_slices()[-1][0]
    blob[w] = np.random.default_rng(1).normal(0.0, 0.05, size=w.stop - w.start)
    return blob


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        inst = _instances(c, seed)
        solver = mpfc.BatchSolver([_params(i) for i in inst])
        return dict(c=c, solver=solver, states=[_state(i, i["seed"])[0] for i in inst])
    if c["kind"] == "train":
        f = _samples(c, seed)
        return dict(c=c, trainer=guess.Trainer(_blob(), c["B"], c["H"], c["W"], lr=2e-3), fields=[f[2], f[1], f[0], f[3]])
    st, W, target, _ = _state(c, seed)
    solver = mpfc.Solver(_params(c))
    if c["pinned"]:
        solver.set_pinning(W, target)
    if c["guess"] == "learned":
        guess.attach(solver, guess.load())
    if c["kind"] == "energy":
        solver.set_state(*st)
    return dict(c=c, solver=solver, state=st)


def _ck(rc):
    if rc != 0:
        raise mpfc.MPFCError(rc, "batch")


def run(state):
    c = state["c"]
    if c["kind"] == "batch":
        # states in and out stay on the device: the C ABI takes host or device pointers
        b, P = state["solver"], lambda t: ctypes.c_void_p(t.data_ptr())
        out = []
        for i, st in enumerate(state["states"]):
            _ck(b.lib.mpfc_batch_set_state(b.h, i, *[P(t) for t in st]))
        b.step(c["scheme"], c["steps"])
        for i, st in enumerate(state["states"]):
            got = [torch.empty_like(t) for t in st]
            _ck(b.lib.mpfc_batch_get_state(b.h, i, *[P(t) for t in got]))
            out.append(got)
        return out
    if c["kind"] == "train":
        tr = state["trainer"]
        tr.train_step(*state["fields"])
        return dict(params=tr.params, grads=tr.grads, yhat=tr.yhat[:, :1])
    solver = state["solver"]
    if c["kind"] == "energy":
        e = solver.energy()
        return dict(F=e["F"], pseudoF=e["pseudoF"], tildeF=e["tildeF"], mass=solver.mass())
    solver.set_state(*state["state"])
    solver.step(c["scheme"], c["steps"])
    return solver.get_state(device=True)


def work(case):
    c = case
    if c["kind"] == "train":
        N = c["B"] * c["H"] * c["W"]
        macs = 9 * (3 * 32 + 3 * 32 * 32 + 32)
        return dict(bytes=N * 4 * 8.0 + 16.0 * guess.PARAM_COUNT, flops=3 * 2.0 * macs * N)
    if c["kind"] == "batch":
        cells = sum(i["m"] * i["n"] for i in _instances(c, 1))
    else:
        cells = c["m"] * c["n"]
    if c["kind"] == "energy":
        return dict(bytes=24.0 * cells, flops=14 * 4 / 3 * 60.0 * cells)
    # state in and out; a V-cycle's sweeps (46 flops per cell and sweep), transfers and residual, four V-cycles a step
    return dict(bytes=48.0 * cells, flops=c["steps"] * 4 * 4 / 3 * (4 * 46 + 60.0) * cells)


# -------------------------------------------------------------------------- exact
def _exact_energy(c, sp, st):
    phi, prev, psi = st
    h2, alpha = c["h"] ** 2, 1.0 - c["epsilon"]
    lam = sp.lam.clone()
    lam[0, 0] = 1.0
    f = sp.fwd(psi - psi.mean()) / -lam
    f[0, 0] = 0.0

    def grad2(a):
        up = torch.cat([a[1:], a[-1:]]) if sp.even else a.roll(-1, 0)
        return float(((a.roll(-1, 1) - a) ** 2 + (up - a) ** 2).sum())

    F = 0.25 * h2 * float((phi ** 4).sum()) + 0.5 * alpha * h2 * float((phi ** 2).sum()) - grad2(phi) + \
        0.5 * h2 * float((sp.lap(phi) ** 2).sum())
    pseudo = F if c["model"] == "pfc" else F + h2 * float((psi * sp.inv(f)).sum()) / (2.0 * c["M"])
    return dict(F=F, pseudoF=pseudo, tildeF=pseudo + 0.5 * grad2(phi - prev), mass=h2 * float(phi.sum()))


def _exact_train(c, seed):
    f = _samples(c, seed)
    blob = torch.from_numpy(np.asarray(_blob(), dtype=np.float64)).to(DEV).requires_grad_(True)
    norm = blob.detach()[:4]
    p2, p1, p0, nx = f
    mean = p0.mean(dim=(1, 2), keepdim=True)
    x = torch.stack([(p0 - mean) / norm[0], (p0 - p1) / norm[1], (p0 - 2 * p1 + p2) / norm[2]], 1)
    y = (nx - 2 * p0 + p1) / norm[3]
    a, off = x, 4
    for l, (ci, co) in enumerate(guess.LAYERS):
        w = blob[off:off + 9 * ci * co].view(3, 3, ci, co).permute(3, 2, 0, 1)
        off += 9 * ci * co
        b = blob[off:off + co]
        off += co
        a = torch.nn.functional.conv2d(torch.nn.functional.pad(a, (1, 1, 1, 1), mode="circular"), w, b)
        if l < 4:
            a = torch.nn.functional.gelu(a)
    loss = ((a[:, 0] - y) ** 2).mean()
    loss.backward()
    g = blob.grad.clone()
    g[:4] = 0.0
    # Adam's first step: m / (1 - b1) = g and v / (1 - b2) = g^2
    new = blob.detach() - 2e-3 * g / (g.abs() + 1e-8)
    new[:4] = norm
    return dict(params=new, grads=g, yhat=a.detach().permute(0, 2, 3, 1).reshape(-1, 1))


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return _exact_train(c, seed)
    if c["kind"] == "batch":
        out = []
        for i in _instances(c, seed):
            st, _, _, sp = _state(i, i["seed"])
            for _ in range(c["steps"]):
                st = sp.step(*st)
            out.append(list(st))
        return out
    st, _, _, sp = _state(c, seed)
    if c["kind"] == "energy":
        return _exact_energy(c, sp, st)
    for _ in range(c["steps"]):
        st = sp.step(*st)
    return list(st)
