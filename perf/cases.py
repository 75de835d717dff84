"""The work a user of this package has it do, as cases that can be timed and compared.

listed() and draw(rng) give cases (dicts of plain values), prepare(case, seed) what a program
has in hand before the call, run(state) one pass through the public entry points, work(case)
the bytes and operations the pass cannot do without, and exact(case, seed) the same outputs in
64-bit torch, written from the method (Lin & Fessler, arXiv 2005.08661) without this package.

Acquisitions follow the recipe of the package's synthetic volumes, drawn on the GPU: an
ellipsoid phantom (semi-axes 0.4 / 0.35 / 0.4 of the grid, magnitude 1 inside and 0.05
outside), a field map that is a sum of random Gaussians, coils on a ring, complex noise at a
stated SNR, and the support mask dilated by two voxels.  Echo times are in ms.

Kinds of case:
  solve    set_data + solve: one acquisition turned into a field map
  cost     set_data was done; one evaluation of cost, gradient and curvature (a program with
           its own optimiser calls this)
  precond  ic_factor + ic_apply at a given map (a program with its own linear solver)
  batch    FieldMapBatch: many volumes of uneven sizes solved together
  wf       the water-fat pipeline: set_data, sweep + PWLS start, solve, amplitudes
  diff     torch.autograd: field_map_solve forward, loss, backward to images and beta
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2005_08661_gb300 as fmpkg
from paper_2005_08661_gb300.autograd import field_map_solve

TE3 = "0,2,10"
TE_WF = "1.2,2.2,3.2,4.2,5.2,6.2"
WORK_MAX = 256 * 256 * 128 * 8  # voxels x coils of the largest listed case
LARGE_NITER = 50


def _case(kind, nx, ny, nz, nc=1, te=TE3, snr=20.0, peak=150.0, beta=0.125, precision="fp32", precond="ic0",
          curvature="literal", niter=0, mask=True, dilate=2, name=None, **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, nc=nc, te=te, snr=snr, peak=peak, beta=beta, precision=precision,
             precond=precond, curvature=curvature, niter=niter, mask=mask, dilate=dilate)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one evaluation of a small slab: launches and latency are all there is
        _case("cost", 64, 64, 16, 1, snr=30.0, name="cost_64x64x16_c1"),
        # a small single-coil slab from images to map: the interactive case
        _case("solve", 64, 64, 16, 1, niter=50, snr=30.0, name="solve_64x64x16_c1"),
        # the same in the library's double precision mode
        _case("solve", 64, 64, 16, 1, precision="fp64", niter=20, snr=30.0, name="solve_64x64x16_c1_fp64"),
        # the paper's phantom scan: few slices, 32 coils, short echo spacings; IC(0), then the
        # incomplete Cholesky with a drop tolerance that the paper prefers
        _case("solve", 74, 74, 10, 32, te="0,1,2.3", niter=20, name="solve_74x74x10_c32"),
        _case("solve", 74, 74, 10, 32, te="0,1,2.3", precond="ict", niter=20, name="solve_74x74x10_c32_ict"),
        # an odd-sized acquisition with four echoes and four coils
        _case("solve", 133, 117, 45, 4, te="0,1.5,4,9.5", niter=30, name="solve_133x117x45_c4_e4"),
        # a whole-head volume, coil-combined curvature (the cheap option)
        _case("solve", 192, 192, 96, 8, curvature="combined", peak=250.0, niter=40, name="solve_192x192x96_c8_comb"),
        # the headline acquisition: a high-resolution volume with eight coils
        _case("solve", 256, 256, 128, 8, snr=15.0, peak=250.0, niter=LARGE_NITER, name="solve_256x256x128_c8"),
        # the preconditioner alone, for a program with its own solver
        _case("precond", 192, 160, 96, 1, peak=250.0, snr=30.0, name="precond_192x160x96"),
        # a study of volumes of uneven sizes, one or eight coils
        _case("batch", 192, 176, 96, 8, volumes=8, niter=20, snr=30.0, name="batch_8_volumes"),
        # water-fat imaging with six echoes
        _case("wf", 192, 192, 64, 1, te=TE_WF, peak=200.0, beta=2.0 ** -7, niter=30, snr=30.0,
              name="water_fat_192x192x64"),
        # differentiating the map: forward solve, loss, backward
        _case("diff", 128, 128, 64, 8, peak=250.0, niter=60, name="diff_128x128x64_c8"),
    ]



def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "cost", "precond", "batch", "wf", "diff"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(nc, limit=WORK_MAX // 2):
        while True:
            nx, ny, nz = size(48, 256), size(48, 256), size(10, 128)
            if nx * ny * nz * nc <= limit:
                return nx, ny, nz

    snr = round(rng.uniform(15.0, 25.0), 1)   # of one coil of an array
    snr1 = round(rng.uniform(28.0, 34.0), 1)  # of images that come as one coil
    beta = rng.choice([2.0 ** -4, 2.0 ** -3, 2.0 ** -2])
    mask = rng.random() < 0.85
    if kind == "solve":
        form = rng.choice(["literal", "literal", "combined", "phantom", "fp64"])
        if form == "phantom":
            nx, ny, nz = size(48, 96), size(48, 96), rng.randint(6, 14)
            return _case("solve", nx, ny, nz, rng.choice([12, 16, 32]), te="0,1,2.3", snr=snr, beta=beta,
                         precond=rng.choice(["ic0", "ict", "diag"]), niter=rng.randint(8, 20), mask=mask)
        if form == "fp64":
            return _case("solve", size(48, 80), size(48, 80), size(10, 20), 1, snr=snr1, beta=beta, precision="fp64",
                         niter=rng.randint(5, 15), mask=mask)
        nc = rng.choice([1, 2, 3, 4, 6, 8, 8])
        te = rng.choice([TE3, TE3, "0,2.5", "0,1.5,4,9.5"])
        nx, ny, nz = grid(nc)
        return _case("solve", nx, ny, nz, nc, te=te, snr=snr1 if nc == 1 else snr, beta=beta, curvature=form,
                     precond=rng.choice(["ic0", "ic0", "ic0", "rb"]), niter=rng.randint(10, 30), mask=mask)
    if kind == "cost":
        nc = rng.choice([1, 2, 4, 8])
        nx, ny, nz = grid(nc)
        return _case("cost", nx, ny, nz, nc, te=rng.choice([TE3, "0,2.5", "0,1.5,4,9.5"]),
                     snr=snr1 if nc == 1 else snr, beta=beta,
                     mask=mask)
    if kind == "precond":
        nx, ny, nz = grid(1)
        return _case("precond", nx, ny, nz, 1, snr=snr1, beta=beta, mask=mask)
    if kind == "batch":
        return _case("batch", size(64, 160), size(64, 160), size(16, 64), rng.choice([1, 8]), snr=snr1, beta=beta,
                     volumes=rng.randint(3, 8), niter=rng.randint(5, 15))
    if kind == "wf":
        return _case("wf", size(64, 192), size(64, 192), size(10, 48), 1, te=TE_WF, snr=snr1, peak=200.0,
                     beta=2.0 ** -7, niter=rng.randint(8, 20), mask=mask)
    return _case("diff", size(64, 128), size(64, 128), size(16, 64), rng.choice([4, 8]), snr=max(snr, 20.0),
                 beta=max(beta, 0.125),
                 niter=rng.randint(30, 60))


# ---------------------------------------------------------------------------- acquisitions

def _te(case):
    return [float(v) for v in case["te"].split(",")]


def _dilate(case):
    """Voxels by which the support mask exceeds the object, or None: no mask, every voxel an unknown."""
    return case["dilate"] if case["mask"] else None


def _axis(n):
    return torch.arange(n, dtype=torch.float64, device="cuda") - (n - 1) / 2.0


def _grids(nx, ny, nz):
    return _axis(nx)[None, None, :], _axis(ny)[None, :, None], _axis(nz)[:, None, None]


def _dilated(inside, r):
    out = inside.clone()
    nz, ny, nx = inside.shape
    pad = torch.zeros((nz + 2 * r, ny + 2 * r, nx + 2 * r), dtype=torch.bool, device="cuda")
    pad[r:r + nz, r:r + ny, r:r + nx] = inside
    for dz in range(-r, r + 1):
        for dy in range(-r, r + 1):
            for dx in range(-r, r + 1):
                if 0 < dx * dx + dy * dy + dz * dz <= r * r:
                    out |= pad[r + dz:r + dz + nz, r + dy:r + dy + ny, r + dx:r + dx + nx]
    return out


def _blobs(rng, nx, ny, nz, n, signed, spread):
    x, y, z = _grids(nx, ny, nz)
    f = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    for _ in range(n):
        while True:
            u = rng.uniform(-1.0, 1.0, size=3)
            if float(u @ u) <= 1.0:
                break
        c = u * np.array([0.4 * nx, 0.35 * ny, 0.4 * nz])
        s = rng.uniform(*spread, size=3) * np.array([nx, ny, nz], dtype=np.float64)
        amp = rng.uniform(0.5, 1.0) * (-1.0 if signed and rng.uniform() < 0.5 else 1.0)
        f += amp * (torch.exp(-0.5 * ((z - c[2]) / s[2]) ** 2) * torch.exp(-0.5 * ((y - c[1]) / s[1]) ** 2)
                    * torch.exp(-0.5 * ((x - c[0]) / s[0]) ** 2))
    return f / f.abs().max()


def _coils(rng, nx, ny, nz, nc):
    x, y, z = _grids(nx, ny, nz)
    rad, sig = 0.6 * nx, 0.35 * nx
    out = []
    for k in range(nc):
        a, ph = 2.0 * math.pi * k / nc, rng.uniform(0.0, 2.0 * math.pi)
        m = (torch.exp(-0.5 * (z / sig) ** 2) * torch.exp(-0.5 * ((y - rad * math.sin(a)) / sig) ** 2)
             * torch.exp(-0.5 * ((x - rad * math.cos(a)) / sig) ** 2))
        out.append(torch.polar(m, torch.full_like(m, ph)))
    return torch.stack(out)


def _fat():
    """A six-peak fat spectrum at 3 T: relative amplitudes and offsets in cycles per ms."""
    ppm = np.array([-3.80, -3.40, -2.60, -1.94, -0.39, 0.60])
    amp = np.array([0.087, 0.694, 0.128, 0.004, 0.039, 0.048])
    return amp / amp.sum(), ppm * 42.577478 * 3.0 / 1000.0


def _acquire(nx, ny, nz, nc, te, snr, peak, precision, dilate, seed, fat=False):
    """One acquisition as a scanner delivers it: images, coil maps, support mask, and the true map."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(rng.integers(1 << 40)))
    x, y, z = _grids(nx, ny, nz)
    inside = (z / (0.4 * nz)) ** 2 + (y / (0.35 * ny)) ** 2 + (x / (0.4 * nx)) ** 2 <= 1.0
    omega = _blobs(rng, nx, ny, nz, 5, True, (0.1, 0.3)) * (peak * 2.0 * math.pi / 1000.0)
    if fat:
        water = torch.where(inside, 0.2 + 0.8 * _blobs(rng, nx, ny, nz, 4, False, (0.15, 0.4)), 0.05)
        fatm = torch.where(inside, _blobs(rng, nx, ny, nz, 4, False, (0.15, 0.4)), 0.0)
        amp, freq = _fat()
    else:
        water, fatm = torch.where(inside, 1.0, 0.05).double(), None
    s = _coils(rng, nx, ny, nz, nc) if nc > 1 else None
    cd = torch.complex64 if precision == "fp32" else torch.complex128
    img = torch.empty((len(te), nc, nz, ny, nx), dtype=cd, device="cuda")
    sq = 0.0
    for l, t in enumerate(te):
        m = water if fatm is None else water + fatm * complex(np.sum(amp * np.exp(2j * math.pi * freq * t)))
        ph = torch.polar(torch.ones_like(omega), omega * t) * m
        for c in range(nc):
            v = ph if s is None else ph * s[c]
            img[l, c] = v.to(cd)
            sq = sq + (v[inside].abs() ** 2).sum()
    sigma = torch.sqrt(sq / (inside.sum() * len(te) * nc)) / (math.sqrt(2.0) * 10.0 ** (snr / 20.0))
    rd = torch.float32 if precision == "fp32" else torch.float64
    for l in range(len(te)):
        for c in range(nc):
            n = torch.randn((nz, ny, nx, 2), dtype=rd, device="cuda", generator=gen)
            img[l, c] += torch.view_as_complex(n * sigma.to(rd))
    mask = None if dilate is None else _dilated(inside, dilate).to(torch.uint8)
    return img, (None if s is None else s.to(cd).contiguous()), mask, omega


def _batch_shapes(case):
    """Uneven volumes up to the case's size: multiples of 16, every other one with one coil."""
    out = []
    for k in range(case["volumes"]):
        f = 1.0 - 0.6 * k / max(case["volumes"] - 1, 1)
        nx, ny, nz = (max(16, int(case[a] * f) // 16 * 16) for a in ("nx", "ny", "nz"))
        out.append((nx, ny, nz, case["nc"] if k % 2 == 0 else 1))
    return out


def prepare(case, seed):
    te = _te(case)
    if case["kind"] == "batch":
        shapes = _batch_shapes(case)
        vols = [_acquire(nx, ny, nz, nc, te, case["snr"], case["peak"], case["precision"], case["dilate"], (seed, k))[:3]
                for k, (nx, ny, nz, nc) in enumerate(shapes)]
        fb = fmpkg.FieldMapBatch([(nx, ny, nz, nc, len(te)) for nx, ny, nz, nc in shapes],
                                 precision=case["precision"])
        fb.set_fraction(0.25)  # what the autotuner settles on for such mixes
        return dict(case=case, te=te, fb=fb, vols=vols)
    img, s, mask, omega = _acquire(case["nx"], case["ny"], case["nz"], case["nc"], te, case["snr"], case["peak"],
                                   case["precision"], _dilate(case), (seed, 0), fat=case["kind"] == "wf")
    fm = fmpkg.FieldMap(case["nx"], case["ny"], case["nz"], ncoil=case["nc"], necho=len(te),
                        precision=case["precision"], precond=case["precond"], curvature=case["curvature"])
    st = dict(case=case, te=te, fm=fm, y=img, s=s, mask=mask)
    rd = torch.float32 if case["precision"] == "fp32" else torch.float64
    if case["kind"] in ("cost", "precond"):
        fm.set_data(img, s, te, mask, case["beta"])
        st["w"] = _trial_map(case, seed, omega).to(rd)
        if case["kind"] == "precond":
            st["g"] = torch.randn(omega.shape, dtype=rd, device="cuda", generator=_gen(seed)) * _mask01(st).to(rd)
    if case["kind"] == "wf":
        amp, freq = _fat()
        fm.set_fat_model(amp, freq)
    if case["kind"] == "diff":
        st["target"] = (omega * _mask01(st)).to(rd)
        st["beta"] = torch.tensor(case["beta"], dtype=torch.float64)
    return st


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(np.random.default_rng((seed, 77)).integers(1 << 40)))
    return g


def _mask01(st):
    return torch.ones(1, device="cuda") if st["mask"] is None else st["mask"].to(torch.float64)


def _trial_map(case, seed, omega):
    """A map part-way through a solve: the truth plus a few Hz of noise."""
    return omega + 0.05 * torch.randn(omega.shape, dtype=torch.float64, device="cuda", generator=_gen(seed + 1))


def run(st):
    case, te = st["case"], st["te"]
    if case["kind"] == "batch":
        fb = st["fb"]
        for k, (y, s, m) in enumerate(st["vols"]):
            fb.set_data(k, y, s, te, m, case["beta"])
        return fb.solve(niter=case["niter"], want_history=False)[0]
    fm = st["fm"]
    if case["kind"] == "cost":
        return fm.cost_grad(st["w"])
    if case["kind"] == "precond":
        ip, p = fm.ic_factor(st["w"]), fm.ic_apply(st["g"])
        return ip, p, (st["g"] * p).sum()  # r'z, which every preconditioned solver takes next
    if case["kind"] == "diff":
        y, b = st["y"].requires_grad_(True), st["beta"].requires_grad_(True)
        y.grad = b.grad = None
        w = field_map_solve(y, b, fm, st["s"], te, st["mask"], niter=case["niter"])
        ((w - st["target"]) ** 2).sum().backward()
        return w.detach(), y.grad, b.grad
    fm.set_data(st["y"], st["s"], te, st["mask"], case["beta"])
    if case["kind"] == "wf":
        w, hist = fm.solve(fm.wf_init(), niter=case["niter"])
        return (w, hist.tolist()) + tuple(fm.wf_amplitudes(w))
    w, hist = fm.solve(niter=case["niter"])
    return w, hist.tolist()  # the costs as ordinary numbers


def _mask_voxels(nx, ny, nz, mask=True):
    """Voxels of the dilated ellipsoid, by its volume."""
    full = nx * ny * nz
    return min(full, 4.0 / 3.0 * math.pi * (0.4 * nx + 2) * (0.35 * ny + 2) * (0.4 * nz + 2)) if mask else full


def work(case):
    """Each input read once, each output written once; the method's own operations (about 12
    per echo pair and evaluation, 14 per wrapped-sinc term of the curvature)."""
    L = len(_te(case))
    P, val = L * (L - 1) // 2, 4 if case["precision"] == "fp32" else 8

    def one(nx, ny, nz, nc, evals, mask=True):
        n, m = nx * ny * nz, _mask_voxels(nx, ny, nz, mask)
        terms = nc * nc if case["curvature"] == "literal" else 1
        return (n * ((L + (nc > 1)) * nc * 2 * val + 1 + val), evals * m * P * (12 + 14 * terms))

    nls, it = 5, case["niter"]
    if case["kind"] == "batch":
        parts = [one(nx, ny, nz, nc, nls * it + 1) for nx, ny, nz, nc in _batch_shapes(case)]
        return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}
    n, m = case["nx"] * case["ny"] * case["nz"], _mask_voxels(case["nx"], case["ny"], case["nz"], case["mask"])
    evals = {"solve": nls * it + 1, "wf": nls * it + 1, "diff": nls * it + 2, "cost": 1, "precond": 1}[case["kind"]]
    b, f = one(case["nx"], case["ny"], case["nz"], case["nc"], evals, case["mask"])
    if case["kind"] == "cost":  # the data are in the handle: pairs and, for several coils, coil weights
        per = P * 2 * val + (L * case["nc"] * 2 * val if case["nc"] > 1 else 0) + val + 1
        return {"bytes": m * per + 2 * n * val, "flops": f}
    if case["kind"] == "precond":
        return {"bytes": m * (P * 2 * val + 1 + 2 * val) + 2 * n * val, "flops": f + 30 * m}
    if case["kind"] == "wf":
        return {"bytes": b + 4 * n * val, "flops": f + 100 * m * P * 12}
    if case["kind"] == "diff":
        return {"bytes": b + n * L * case["nc"] * 2 * val, "flops": f}
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------- 64-bit values

class _Ref:
    """The method in 64-bit torch: data term, IC(0) and the NCG iteration on one acquisition."""

    def __init__(self, case, y, s, mask):
        nz, ny, nx = y.shape[2:]
        self.shape, self.dev = (nz, ny, nx), y.device
        self.beta, self.te = case["beta"], _te(case)
        self.literal = case["curvature"] == "literal" and y.shape[1] > 1
        m = torch.ones(self.shape, dtype=torch.bool, device="cuda") if mask is None else mask != 0
        pad = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=torch.bool, device="cuda")
        pad[1:-1, 1:-1, 1:-1] = m
        self.m = m
        self.idx = pad.reshape(-1).nonzero()[:, 0]  # mask voxels in the padded grid, natural order
        self.nbr = [1, nx + 2, (nx + 2) * (ny + 2)]
        self.npad = pad.numel()
        flat = pad.reshape(-1).double()
        self.edges = [flat[self.idx + o] for o in self.nbr]          # in-mask +x, +y, +z neighbour
        self.lower = [flat[self.idx - o] for o in self.nbr]
        self.count = sum(self.edges) + sum(self.lower)
        L, C = y.shape[0], y.shape[1]
        Y = y[:, :, m].to(torch.complex128)
        S = torch.ones((C, Y.shape[2]), device="cuda") if s is None else s[:, m]
        S = S.to(torch.complex128)
        nrm = (S.abs() ** 2).sum(0)
        W = S.conj()[None] * Y / torch.sqrt(L * torch.where(nrm > 0, nrm, 1.0)) * (nrm > 0)
        self.A, self.psi = W.abs(), W.angle()
        Z = W.sum(1)
        self.pairs = []
        for a in range(L):
            for b in range(a + 1, L):
                R = Z[a].conj() * Z[b]
                self.pairs.append((a, b, self.te[a] - self.te[b], R.abs(), R.angle()))
        self.K = ((self.A.sum(1).sum(0)) ** 2 - Z.abs().sum(0) ** 2).sum()
        e = (Z[0].conj() * Z[1]).angle()
        self.w0 = e / (self.te[1] - self.te[0])

    def full(self, v):
        out = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        out[self.m] = v
        return out

    def _spread(self, v):
        f = torch.zeros(self.npad, dtype=torch.float64, device="cuda")
        f[self.idx] = v
        return f

    @staticmethod
    def _sinc(u):
        u = u - 2.0 * math.pi * torch.round(u / (2.0 * math.pi))
        return torch.where(u == 0, 1.0, torch.sin(u) / torch.where(u == 0, 1.0, u))

    def data(self, w):
        cost, grad, curv = self.K.clone(), torch.zeros_like(w), torch.zeros_like(w)
        for a, b, dt, R, ang in self.pairs:
            th = ang + w * dt
            cost = cost + 4.0 * (R * torch.sin(th / 2) ** 2).sum()
            grad += 2.0 * dt * R * torch.sin(th)
            if self.literal:
                for c in range(self.A.shape[1]):
                    for d in range(self.A.shape[1]):
                        curv += 2.0 * dt * dt * self.A[a, c] * self.A[b, d] * self._sinc(
                            self.psi[b, d] - self.psi[a, c] + w * dt)
            else:
                curv += 2.0 * dt * dt * R * self._sinc(th)
        return cost, grad, curv

    def diffs(self, v):
        f = self._spread(v)
        return [e * (f[self.idx + o] - v) for e, o in zip(self.edges, self.nbr)]

    def cost_grad(self, w):
        cost, g, d = self.data(w)
        f = self._spread(w)
        lap = self.count * w
        for o in self.nbr:
            lap = lap - f[self.idx + o] - f[self.idx - o]
        reg = sum((e ** 2).sum() for e in self.diffs(w))
        return cost + 0.5 * self.beta * reg, g + self.beta * lap, d

    def planes(self):
        """Mask voxels by hyperplane x + y + z, as positions in the list and in the padded grid."""
        if not hasattr(self, "_planes"):
            px, py = self.nbr[1], self.nbr[2] // self.nbr[1]
            t = self.idx % px + (self.idx // px) % py + self.idx // (px * py)
            order = torch.argsort(t, stable=True)
            cnt = torch.bincount(t).tolist()
            self._planes, at = [], 0
            for n in cnt:
                if n:
                    self._planes.append((order[at:at + n], self.idx[order[at:at + n]]))
                at += n
        return self._planes

    def ic(self, d, g=None):
        """(1/pi, (L L')^-1 g): pivots and substitutions of the zero-fill incomplete Cholesky."""
        H = d + self.beta * self.count
        ip = torch.zeros(self.npad, dtype=torch.float64, device="cuda")
        v = torch.zeros_like(ip)
        x, y, z = self.nbr
        for k, j in self.planes():
            r = 1.0 / (H[k] - self.beta ** 2 * (ip[j - x] + ip[j - y] + ip[j - z]))
            ip[j] = r
            if g is not None:
                v[j] = r * (g[k] + self.beta * (v[j - x] + v[j - y] + v[j - z]))
        if g is None:
            return ip[self.idx], None
        p = torch.zeros_like(ip)
        for k, j in reversed(self.planes()):
            p[j] = v[j] + self.beta * ip[j] * (p[j + x] + p[j + y] + p[j + z])
        return ip[self.idx], p[self.idx]

    def solve(self, niter, precond, nls=5):
        w, z, hist = self.w0.clone(), None, []
        gp_prev = g_prev = None
        for it in range(niter + 1):
            cost, g, d = self.cost_grad(w)
            hist.append(cost)
            if it == niter:
                return w, torch.stack(hist)
            p = self.ic(d, g)[1] if precond == "ic0" else g / (d + self.beta * self.count) if precond == "diag" else g
            mu = 0.0 if it == 0 else ((g - g_prev) * p).sum() / gp_prev
            z = -p if it == 0 else -p + mu * z
            cz, cw = self.diffs(z), self.diffs(w)
            cz2, czw = sum((e ** 2).sum() for e in cz), sum((e * f).sum() for e, f in zip(cz, cw))
            alpha = -(z * g).sum() / ((z * z * d).sum() + self.beta * cz2)
            for _ in range(1, nls):
                _, gr, cu = self.data(w + alpha * z)
                slope = (z * gr).sum() + self.beta * (czw + alpha * cz2)
                alpha = alpha - slope / ((z * z * cu).sum() + self.beta * cz2)
            w = w + alpha * z
            gp_prev, g_prev = (g * p).sum(), g


def exact(case, seed):
    te = _te(case)
    terms = case["nc"] ** 2 if case["curvature"] == "literal" else 1
    m = _mask_voxels(case["nx"], case["ny"], case["nz"], case["mask"])
    if case["kind"] not in ("cost", "precond", "solve") or case["precond"] not in ("ic0", "diag", "none"):
        return None
    steps = (case["nx"] + case["ny"] + case["nz"]) * 2 * case["niter"]
    if case["kind"] == "solve" and (m * terms * (5 * case["niter"] + 1) * len(te) > 3e9 or steps > 40000):
        return None  # far over the seconds that are wanted
    img, s, mask, omega = _acquire(case["nx"], case["ny"], case["nz"], case["nc"], te, case["snr"], case["peak"],
                                   case["precision"], _dilate(case), (seed, 0))
    ref = _Ref(case, img, s, mask)
    if case["kind"] == "solve":
        w, hist = ref.solve(case["niter"], case["precond"])
        return ref.full(w), hist.tolist()
    rd = torch.float32 if case["precision"] == "fp32" else torch.float64
    w = _trial_map(case, seed, omega).to(rd).double()[ref.m]
    if case["kind"] == "cost":
        cost, g, d = ref.cost_grad(w)
        return float(cost), ref.full(g), ref.full(d)
    g = torch.randn(omega.shape, dtype=rd, device="cuda", generator=_gen(seed)).double()[ref.m]
    ip, p = ref.ic(ref.data(w)[2], g)
    return ref.full(ip), ref.full(p), (g * p).sum()
