"""The work that a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the public Python entry points (``Slit``, ``Ensemble``,
``MLP``) with the options a program would pass and default launch shapes. Five
kinds:

  slit       advance a slit or a periodic box and read the density and the
             velocity into device buffers the caller owns (with or without the
             attractive tail, FP32 or FP16 populations, one or two buffers)
  evaluate   set given fields and read pressure, forces and the FP64 profiles
  ensemble   advance many slits of uneven widths between two residual checks
             and read the fields
  forward    the warm-start network on a batch of slit parameters
  train      a few Adam steps of that network, then its weights

``exact`` restates the method in 64 bits with plain torch operations.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

KT = 1.0 / 3.0
C = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
     (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1))
HMAX = 80  # planes of the widest slit the network predicts


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _slit(nx, ny, nz, sigma, eta, tau, body, steps, **kw):
    c = dict(kind="slit", nx=nx, ny=ny, nz=nz, sigma=sigma, eta=eta, tau=tau, body=body, steps=steps,
             periodic_z=False, storage=0, inplace=False, shifted=False, g2_form=0, tail=False, eps=0.0)
    c.update(kw)
    return c


def _ensemble(slits, nx, ny, storage, inplace, steps):
    return dict(kind="ensemble", slits=slits, nx=nx, ny=ny, sigma=4, storage=storage, inplace=inplace, steps=steps)


def listed():
    return [
        # the smallest slit (the parity workload): 100 steps between two looks
        # at the fields; latency and launches
        dict(_slit(16, 16, 32, 4, 0.25, 1.0, 1e-6, 100), name="slit_16x16x32"),
        # an ordinary slit, narrower than a warp-wide force tile
        dict(_slit(64, 64, 128, 8, 0.25, 0.8, 1e-6, 20), name="slit_64x64x128"),
        # odd extents and a diameter without a specialised force kernel
        dict(_slit(203, 117, 75, 6, 0.22, 0.9, 1e-6, 10), name="slit_203x117x75_ragged"),
        # the benchmark's slit: 10 steps between two looks, FP32 populations
        dict(_slit(512, 512, 192, 12, 0.25, 0.7, 5e-7, 10), name="slit_512x512x192"),
        # the same slit with FP16 populations (half of the population memory)
        dict(_slit(512, 512, 192, 12, 0.25, 0.7, 5e-7, 10, storage=1), name="slit_512x512x192_f16"),
        # a Lennard-Jones tail on power-of-two extents (spectral sum)
        dict(_slit(256, 256, 128, 8, 0.25, 0.8, 1e-6, 10, tail=True, eps=0.3), name="slit_tail_256x256x128"),
        # the same model on extents that are no powers of two (direct sum)
        dict(_slit(60, 52, 40, 4, 0.25, 0.8, 1e-6, 10, tail=True, eps=0.3), name="slit_tail_60x52x40_ragged"),
        # the functional alone: pressure, forces and profiles of given fields
        dict(kind="evaluate", nx=256, ny=192, nz=96, sigma=8, eta=0.25, g2_form=0, name="evaluate_256x192x96"),
        # 256 slits of 32 x 32 x H, FP16 in place: one residual check's worth
        dict(_ensemble(256, 32, 32, 1, True, 100), name="ensemble_256_f16"),
        # thin slits that generate the network's training profiles
        dict(_ensemble(2048, 4, 4, 0, True, 100), name="ensemble_2048_thin"),
        # the network on a batch of slit parameters
        dict(kind="forward", rows=65536, name="network_forward_65536"),
        # minibatch training: four steps of the trainer's default batch
        dict(kind="train", rows=1024, steps=4, name="network_train_1024"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["slit"] * 5 + ["tail"] * 2 + ["evaluate", "ensemble", "ensemble", "thin", "forward", "train"])
    if kind == "forward":
        return dict(kind="forward", rows=_log_int(rng, 1, 65536))
    if kind == "train":
        return dict(kind="train", rows=_log_int(rng, 32, 4096), steps=rng.randint(1, 4))
    if kind == "ensemble":
        return _ensemble(_log_int(rng, 8, 256), rng.choice([32, 32, 48, 33]), rng.choice([32, 32, 24, 35]),
                         rng.choice([0, 1]), rng.choice([True, True, False]), 2 * rng.randint(5, 40))
    if kind == "thin":
        return _ensemble(_log_int(rng, 64, 4096), rng.choice([4, 4, 8, 5]), rng.choice([4, 4, 3]), 0, True,
                         2 * rng.randint(10, 50))
    sigma = rng.choice([4, 4, 6, 8, 10, 12])
    if kind == "evaluate":
        return dict(kind="evaluate", nx=_log_int(rng, 6, 300), ny=_log_int(rng, 6, 300), nz=rng.randint(12, 160),
                    sigma=sigma, eta=rng.uniform(0.10, 0.25), g2_form=rng.choice([0, 1]))
    c = _slit(0, 0, 0, sigma, rng.uniform(0.10, 0.22), rng.uniform(0.65, 1.1), 10.0 ** rng.uniform(-7.0, -5.0), 0,
              storage=rng.choice([0, 0, 1]), inplace=rng.choice([False, False, True]))
    if kind == "tail":
        c["sigma"] = rng.choice([4, 4, 6, 8])
        c.update(tail=True, eps=rng.uniform(0.1, 0.3), steps=rng.randint(1, 6))
        if rng.random() < 0.5:
            c.update(nx=rng.choice([32, 64, 128, 256]), ny=rng.choice([32, 64, 128, 256]), nz=rng.randint(20, 128))
        else:
            # the direct sum visits every displacement: bounded by the product
            c.update(nx=_log_int(rng, 20, 100), ny=_log_int(rng, 20, 100), nz=rng.randint(20, 60))
            if c["sigma"] == 8:
                c.update(steps=1)
        return c
    c.update(nx=_log_int(rng, 4, 400), ny=_log_int(rng, 4, 300), nz=rng.randint(14, 192))
    most = int(1e8 / (c["nx"] * c["ny"] * c["nz"]))
    c.update(steps=rng.randint(2, max(3, min(40, most))),
             periodic_z=rng.random() < 0.25, shifted=rng.random() < 0.2, g2_form=rng.choice([0, 0, 1]))
    return c


# ---------------------------------------------------------------------------
# inputs and one pass
# ---------------------------------------------------------------------------
def _n0(eta, sigma):
    return 6.0 * eta / (math.pi * sigma ** 3)


def _slits(case, seed):
    """Widths (the case's), packing fractions, forces and relaxation times (the seed's) of an ensemble."""
    ns, s = case["slits"], case["sigma"]
    H = np.random.default_rng(3).integers(2 * s, 20 * s + 1, ns).astype(np.int32)
    g = np.random.default_rng(seed)
    return H, g.uniform(0.10, 0.25, ns), 10.0 ** g.uniform(-7.0, -5.0, ns), g.uniform(0.6, 1.2, ns)


def _given_fields(case, seed, device):
    """Positive density and small velocity fields that vary over a few spacings."""
    g = torch.Generator(device="cpu").manual_seed(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    z, y, x = (torch.arange(n, dtype=torch.float64) for n in shape)
    out = []
    for amp in (0.10, 0.02, 0.02, 0.05):
        a = torch.zeros(shape, dtype=torch.float64, device=device)
        for _ in range(4):
            k = torch.randint(1, 5, (3,), generator=g)
            ph = torch.rand(3, generator=g, dtype=torch.float64) * 2 * math.pi
            w = [torch.cos(2 * math.pi * int(k[i]) * v / n + ph[i]).to(device)
                 for i, (v, n) in enumerate(zip((z, y, x), shape))]
            a += 0.25 * amp * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
        out.append(a)
    rho = (_n0(case["eta"], case["sigma"]) * (1.0 + out[0])).float().contiguous()
    return rho, torch.stack(out[1:]).float().contiguous()


def _network_inputs(case, seed):
    """Parameters of the 4 -> 3 x 256 -> 160 network, scaled inputs, targets and masks."""
    g = np.random.default_rng(seed)
    dims = [4, 256, 256, 256, 2 * HMAX]
    p = []
    for i, o in zip(dims[:-1], dims[1:]):
        a = math.sqrt(3.0 / i)
        p += [g.uniform(-a, a, o * i), g.uniform(-0.1, 0.1, o)]
    rows = case["rows"] * case.get("steps", 1)
    X = g.standard_normal((rows, 4)).astype(np.float32)
    half = (g.integers(8, HMAX + 1, rows)[:, None] + 1) // 2
    j = np.arange(HMAX)[None, :]
    m = (j < half).astype(np.float32)
    M = np.concatenate([m, m], axis=1)
    d = (j + 0.5) / half
    T = np.concatenate([1.0 + 0.3 * np.tanh(X[:, :1]) * np.exp(-2.0 * d), d * (2.0 - d) * (1.0 + 0.1 * X[:, 1:2])], axis=1)
    return np.concatenate(p).astype(np.float32), X, (T * M).astype(np.float32), M


def prepare(case, seed):
    from paper_0712_2247_gb300 import lbif

    s = dict(kind=case["kind"], case=case)
    if case["kind"] in ("forward", "train"):
        from paper_0712_2247_gb300.mlp import MLP

        p, X, T, M = _network_inputs(case, seed)
        s["net"] = MLP(4, 256, 3, 2 * HMAX, max_batch=case["rows"])
        s["net"].set_params(p)
        s["X"] = torch.from_numpy(X).cuda()
        if case["kind"] == "train":
            s["T"], s["M"] = torch.from_numpy(T).cuda(), torch.from_numpy(M).cuda()
        return s
    if case["kind"] == "ensemble":
        H, eta, F, tau = _slits(case, seed)
        s["g"] = lbif.Ensemble(H, eta, F, tau, case["sigma"], case["nx"], case["ny"], storage=case["storage"],
                               inplace=case["inplace"], seed=seed)
    elif case["kind"] == "evaluate":
        s["g"] = lbif.Slit(case["nx"], case["ny"], case["nz"], case["sigma"], case["eta"], 0.8,
                           g2_form=case["g2_form"])
        s["fields"] = _given_fields(case, seed, "cuda")
        s["p"] = torch.empty(s["g"].shape, device="cuda")
        s["F"] = torch.empty((3,) + s["g"].shape, device="cuda")
        return s
    else:
        s["g"] = lbif.Slit(case["nx"], case["ny"], case["nz"], case["sigma"], case["eta"], case["tau"],
                           periodic_z=case["periodic_z"], body=(case["body"], 0.0, 0.0), g2_form=case["g2_form"],
                           tail=case["tail"], eps=case["eps"], rcut=2.5, storage=case["storage"], seed=seed,
                           inplace=case["inplace"], shifted=case["shifted"])
    s["rho"] = torch.empty(s["g"].shape, device="cuda")
    s["u"] = torch.empty((3,) + s["g"].shape, device="cuda")
    return s


def run(s):
    case = s["case"]
    if s["kind"] == "forward":
        return s["net"].forward(s["X"])
    if s["kind"] == "train":
        b = case["rows"]
        losses = [s["net"].train_step(s["X"][k * b:(k + 1) * b], s["T"][k * b:(k + 1) * b], s["M"][k * b:(k + 1) * b],
                                      lr=1e-3) for k in range(case["steps"])]
        return {"losses": losses, "params": s["net"].get_params()}
    g = s["g"]
    if s["kind"] == "evaluate":
        g.set_fields(*s["fields"])
        g.moments(pressure=s["p"])
        g.forces(out=s["F"])
        n, ux, total = g.profiles()
        return {"p": s["p"], "F": s["F"], "n_z": n, "ux_z": ux, "total": total}
    if s["kind"] == "ensemble":
        # the first call also takes two steps outside the captured graph
        taken = g.run(tol=1e-30, max_steps=case["steps"], check_every=case["steps"])
        g.moments(rho=s["rho"], u=s["u"])
        return {"taken": taken, "rho": s["rho"], "u": s["u"]}
    g.step(case["steps"])
    g.moments(rho=s["rho"], u=s["u"])
    return {"rho": s["rho"], "u": s["u"]}


def work(case):
    """Bytes: populations in and out once a step, density and velocity written
    and read once a step, outputs written. Operations: collision and moments,
    the 18-point rule, the ball sums by rows and discs, the tail as transforms."""
    if case["kind"] in ("forward", "train"):
        par = 4 * 256 + 2 * 256 * 256 + 256 * 160
        if case["kind"] == "forward":
            return {"bytes": case["rows"] * (4 + 160) * 4 + par * 2, "flops": 2.0 * par * case["rows"]}
        return {"bytes": case["steps"] * (case["rows"] * (4 + 2 * 160) * 4 + par * 28),
                "flops": 6.0 * par * case["rows"] * case["steps"]}
    R = case["sigma"] // 2
    if case["kind"] == "evaluate":
        N = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": N * 32.0, "flops": N * (700.0 + 4 * R * R)}
    if case["kind"] == "ensemble":
        N = float(_slits(case, 0)[0].sum()) * case["nx"] * case["ny"]
    else:
        N = float(case["nx"] * case["ny"] * case["nz"])
    per = 2 * 19 * (2 if case["storage"] else 4) + 32
    ops = 850.0 + 4 * R * R
    if case.get("tail"):
        D = int(math.ceil(2.5 * case["sigma"]))
        ops += 12.5 * math.log2(case["nx"] * case["ny"]) + 12 * (2 * D + 1)
    return {"bytes": N * (case["steps"] * per + 16), "flops": N * case["steps"] * ops}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _erf_gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _exact_network(case, seed):
    p, X, T, M = _network_inputs(case, seed)
    dims = [4, 256, 256, 256, 2 * HMAX]
    W, at = [], 0
    for i, o in zip(dims[:-1], dims[1:]):
        for shape in ((o, i), (o,)):
            n = int(np.prod(shape))
            W.append(torch.from_numpy(p[at:at + n]).cuda().double().reshape(shape).requires_grad_(case["kind"] == "train"))
            at += n
    X, T, M = (torch.from_numpy(a).cuda().double() for a in (X, T, M))

    def net(x):
        for k in range(0, len(W), 2):
            x = x @ W[k].T + W[k + 1]
            if k + 2 < len(W):
                x = _erf_gelu(x)
        return x

    if case["kind"] == "forward":
        return net(X)
    m = [torch.zeros_like(w) for w in W]
    v = [torch.zeros_like(w) for w in W]
    losses, b = [], case["rows"]
    for t in range(1, case["steps"] + 1):
        s = slice((t - 1) * b, t * b)
        loss = (M[s] * (net(X[s]) - T[s]) ** 2).sum() / M[s].sum()
        losses.append(float(loss))
        for w, g, a, q in zip(W, torch.autograd.grad(loss, W), m, v):
            a.mul_(0.9).add_(0.1 * g)
            q.mul_(0.999).add_(0.001 * g * g)
            with torch.no_grad():
                w -= 1e-3 * (a / (1 - 0.9 ** t)) / ((q / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"losses": losses, "params": torch.cat([w.detach().reshape(-1) for w in W])}


def _splitmix64(x):
    """The published generator on int64 tensors (wrapping products, logical shifts)."""
    def i64(v):
        return v - (1 << 64) if v >= 1 << 63 else v

    def shr(a, k):
        return (a >> k) & ((1 << (64 - k)) - 1)

    z = x + i64(0x9E3779B97F4A7C15)
    z = (z ^ shr(z, 30)) * i64(0xBF58476D1CE4E5B9)
    z = (z ^ shr(z, 27)) * i64(0x94D049BB133111EB)
    return z ^ shr(z, 31)


class _Exact:
    """The method on a stack of slits along z (one slit, or many with planes
    outside the fluid between them), fields as (nz, ny, nx) doubles."""

    def __init__(self, nx, ny, sigma, H, eta, tau, body, *, gap=0, periodic=False, g2_form=0, tail=False, eps=0.0,
                 shifted=False, dev="cuda"):
        self.sigma, self.periodic, self.g2_form, self.shifted, self.dev = sigma, periodic, g2_form, shifted, dev
        nz = int(sum(H)) + gap * (len(H) - 1)
        self.shape = (nz, ny, nx)
        col = {k: np.zeros(nz) for k in ("fluid", "n0", "om", "body", "wall")}
        z0 = 0
        for h, e, t, b in zip(H, eta, tau, body):
            s = slice(z0, z0 + int(h))
            col["fluid"][s], col["n0"][s], col["om"][s], col["body"][s] = 1.0, _n0(e, sigma), 1.0 / t, b
            j = np.arange(int(h))
            col["wall"][s] = np.minimum(j + 0.5, h - 0.5 - j)
            z0 += int(h) + gap
        self.fluid, self.n0, self.om, self.body, wall = (
            torch.from_numpy(col[k]).to(dev)[:, None, None] for k in ("fluid", "n0", "om", "body", "wall"))
        kappa = 2.0 / (math.sqrt(KT) * math.sqrt(math.pi))
        self.lk = kappa * (torch.ones_like(wall) if periodic else 1.0 - torch.exp(-wall / sigma))
        R = sigma // 2
        ball = [(dz, dy, dx, 1.0) for dz in range(-R, R + 1) for dy in range(-R, R + 1) for dx in range(-R, R + 1)
                if dz * dz + dy * dy + dx * dx <= R * R]
        self.ball = self._transform([(z, y, x, 1.0 / len(ball)) for z, y, x, _ in ball], R)
        self.tail = None
        if tail:
            rmax = 2.5 * sigma
            D = int(math.ceil(rmax))
            d = np.arange(-D, D + 1)
            dz, dy, dx = (a.ravel() for a in np.meshgrid(d, d, d, indexing="ij"))
            r2 = (dx * dx + dy * dy + dz * dz).astype(float)
            ok = (r2 >= sigma ** 2) & (r2 <= rmax ** 2)
            dz, dy, dx, r = dz[ok], dy[ok], dx[ok], np.sqrt(r2[ok])
            k = 4.0 * eps * (-12.0 * sigma ** 12 / r ** 13 + 6.0 * sigma ** 6 / r ** 7) / r
            self.tail = [self._transform((dz, dy, dx, k * c), D) for c in (dx, dy, dz)]

    def _transform(self, taps, reach):
        """Transform of sum_d w_d a(r + d), z padded with zeros against wrapping unless periodic."""
        nz, ny, nx = self.shape
        pz = nz if self.periodic else nz + reach
        if isinstance(taps, list):
            taps = tuple(np.array(t) for t in zip(*taps))
        dz, dy, dx, w = taps
        k = np.zeros((pz, ny, nx))
        np.add.at(k, ((-dz) % pz, (-dy) % ny, (-dx) % nx), w)
        return torch.fft.rfftn(torch.from_numpy(k).to(self.dev)), pz

    def _correlate(self, a, transform):
        k, pz = transform
        nz, ny, nx = self.shape
        return torch.fft.irfftn(torch.fft.rfftn(a, s=(pz, ny, nx)) * k, s=(pz, ny, nx))[:nz]

    def at(self, a, dz, dy, dx):
        """a(r + d), zero beyond the walls."""
        a = torch.roll(a, (-dy, -dx), (1, 2)) if dy or dx else a
        if dz == 0:
            return a
        if self.periodic:
            return torch.roll(a, -dz, 0)
        out = torch.zeros_like(a)
        if abs(dz) < a.shape[0]:
            if dz > 0:
                out[:-dz] = a[dz:]
            else:
                out[-dz:] = a[:dz]
        return out

    def noise(self, seed, amp=1e-3):
        nz, ny, nx = self.shape
        idx = torch.arange(nz * ny * nx, dtype=torch.int64, device=self.dev) ^ seed
        U = ((_splitmix64(idx) >> 11) & ((1 << 53) - 1)).double() / 9007199254740992.0
        return self.fluid * self.n0 * (1.0 + amp * (2.0 * U - 1.0)).reshape(self.shape)

    def g2(self, n):
        e = math.pi * self.sigma ** 3 / 6.0 * self._correlate(n, self.ball)
        num = 1.0 - 0.5 * e + (0.25 * e * e if self.g2_form == 0 else 0.0)
        return num / (1.0 - e) ** 3

    def shell(self, n, u):
        """Force density of Eq. LBHS and the static collisional pressure."""
        s, G = self.sigma, self.g2(n)
        pref = KT * s * s * 4.0 * math.pi
        F = [torch.zeros_like(n) for _ in range(3)]
        P = torch.zeros_like(n)

        def point(d, w):
            a = 1.0 / math.sqrt(sum(c * c for c in d))
            dirs = [c * a for c in d]
            nb, md = self._corners([s * c for c in dirs]), self._corners([0.5 * s * c for c in dirs])
            nq = sum(c * self.at(n, *o) for o, c in nb)
            t = w * sum(c * self.at(G, *o) for o, c in md) * nq
            P.add_(t)
            du = torch.zeros_like(n)
            for c, ua in zip(dirs, u):
                if c:
                    du += c * (sum(k * self.at(ua, *o) for o, k in nb) - ua)
            t *= 1.0 - self.lk * du
            for c, f in zip(dirs, F):
                if c:
                    f.add_(c * t)

        for a in range(3):
            for sa in (1, -1):
                point([sa if k == a else 0 for k in range(3)], 1.0 / 30.0)
        for a, b in ((0, 1), (0, 2), (1, 2)):
            for sa in (1, -1):
                for sb in (1, -1):
                    d = [0, 0, 0]
                    d[a], d[b] = sa, sb
                    point(d, 1.0 / 15.0)
        return [-pref * n * f for f in F], KT * s ** 3 / 6.0 * 4.0 * math.pi * n * P

    @staticmethod
    def _corners(p):
        """Lattice corners (dz, dy, dx) and weights of a point at offset p = (x, y, z)."""
        axes = []
        for v in p:
            lo = math.floor(v + 1e-9)
            t = v - lo
            axes.append([(lo, 1.0)] if abs(t) < 1e-9 else [(lo, 1.0 - t), (lo + 1, t)])
        return [((z, y, x), wx * wy * wz) for x, wx in axes[0] for y, wy in axes[1] for z, wz in axes[2]]

    def force(self, n, u):
        F, _ = self.shell(n, u)
        F[0] += n * self.body
        if self.tail:
            for f, k in zip(F, self.tail):
                f += n * self._correlate(n, k)
        return F

    def _cdot(self, i, v):
        out = 0.0
        for c, a in zip(C[i], v):
            if c:
                out = out + c * a
        return out

    def equilibrium(self, i, n, u, uu):
        w = 1.0 / 3.0 if i == 0 else (1.0 / 18.0 if i < 7 else 1.0 / 36.0)
        cu = self._cdot(i, u)
        return w * n * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)

    def step(self, f, n, u):
        F = self.force(n, u)
        safe = torch.where(self.fluid > 0, n, torch.ones_like(n))
        v = [ua + 0.5 * Fa / safe for ua, Fa in zip(u, F)] if self.shifted else u
        vv = sum(a * a for a in v)
        vF = sum(a * b for a, b in zip(v, F)) if self.shifted else None
        for i in range(19):
            w = 1.0 / 3.0 if i == 0 else (1.0 / 18.0 if i < 7 else 1.0 / 36.0)
            cF = self._cdot(i, F)
            S = 3.0 * w * cF
            if self.shifted:
                S = (1.0 - 0.5 * self.om) * w * (3.0 * (cF - vF) + 9.0 * self._cdot(i, v) * cF)
            f[i] = f[i] - self.om * (f[i] - self.equilibrium(i, n, v, vv)) + S
        out = [f[0]]
        for i in range(1, 19):
            opp = i + 1 if i % 2 else i - 1
            back = [-C[i][2], -C[i][1], -C[i][0]]
            g = self.at(f[i], *back)
            if C[i][2] and not self.periodic:
                src = self.at(self.fluid, back[0], 0, 0)
                g = torch.where((src > 0) | (self.fluid == 0), g, f[opp])
            out.append(g * self.fluid)
        return out

    def moments(self, f):
        n = sum(f)
        safe = torch.where(self.fluid > 0, n, torch.ones_like(n))
        return n, [sum(C[i][a] * f[i] for i in range(19) if C[i][a]) / safe for a in range(3)]

    def advance(self, n, steps):
        u = [torch.zeros_like(n) for _ in range(3)]
        uu = torch.zeros_like(n)
        f = [self.equilibrium(i, n, u, uu) for i in range(19)]
        for _ in range(steps):
            f = self.step(f, n, u)
            n, u = self.moments(f)
        return n, torch.stack(u)


def exact(case, seed):
    if case["kind"] in ("forward", "train"):
        return _exact_network(case, seed)
    if case["kind"] == "ensemble":
        H, eta, F, tau = _slits(case, seed)
        m = _Exact(case["nx"], case["ny"], case["sigma"], H, eta, tau, F, gap=(case["sigma"] + 3) // 4 * 4)
        # the first call builds its graph, which takes two steps besides
        n, u = m.advance(m.noise(seed), case["steps"] + 2)
        return {"taken": None, "rho": n, "u": u}
    kw = dict(g2_form=case["g2_form"])
    if case["kind"] == "evaluate":
        m = _Exact(case["nx"], case["ny"], case["sigma"], [case["nz"]], [case["eta"]], [0.8], [0.0], **kw)
        rho, u = (a.double() for a in _given_fields(case, seed, "cuda"))
        F, pc = m.shell(rho, list(u))
        total = torch.stack([rho.sum()] + [(rho * u[a]).sum() for a in range(3)])
        return {"p": KT * rho + pc, "F": torch.stack(F) / _n0(case["eta"], case["sigma"]),
                "n_z": rho.mean((1, 2)), "ux_z": u[0].mean((1, 2)), "total": total}
    m = _Exact(case["nx"], case["ny"], case["sigma"], [case["nz"]], [case["eta"]], [case["tau"]], [case["body"]],
               periodic=case["periodic_z"], tail=case["tail"], eps=case["eps"], shifted=case["shifted"], **kw)
    n, u = m.advance(m.noise(seed), case["steps"])
    return {"rho": n, "u": u}
