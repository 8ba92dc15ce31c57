"""What a user of this framework has it do, as cases that can be timed and compared.

Four kinds of work, each through the package's public entry points:

- "step":    Adam iterations of a running fit (resumed from a checkpoint), then the parameters:
             the inner loop of every fit;
- "grad":    objective and gradient through `PrismLoss`, for a program with its own optimiser;
- "noalloc": the allocation-free objective and gradient of the C-ABI;
- "review":  a whole call on a new volume with the parameters of an earlier fit: set-up as
             overlapping slabs, objective and predicted signal, stitched whole-volume maps.

A case's volumes are ellipsoid or full masks with smooth two-fiber anatomy, shells of gradient
directions, and Rician noise. Adam's moments in a "step" case are those of a fit under way
(second moments well away from zero), as a resumed fit has them.
"""
import ctypes
import math
import struct

import numpy as np
import torch

import paper_2604_00250_gb300 as prism
from paper_2604_00250_gb300 import _lib

D_CSF, D_GM, D_RES, D_PAR, D_PERP = 3.0e-3, 0.9e-3, 0.2e-3, 1.7e-3, 0.4e-3
B0_MAX = 50.0
STEP0 = 200      # iterations the resumed fits have behind them


class Volume:
    """What `prism.Fitter` takes: mask, signal rows, b-values, b-vectors, optional start."""

    def __init__(self, mask, signal, bvals, bvecs, init=None):
        self.mask, self.signal, self.bvals, self.bvecs, self.init = mask, signal, bvals, bvecs, init


# -- cases ---------------------------------------------------------------------------------------
def _case(kind, shape, **kw):
    c = dict(kind=kind, nx=shape[0], ny=shape[1], nz=shape[2], vols=1, unlike=False, mask="full", n_meas=96, b0=6,
             shells=3, bmax=3000.0, mixed=False, snr=30.0, K=3, loss="mse", cal=False, spatial=False, conn=6, patch=16,
             iters=16)
    c.update(kw)
    return c


def listed():
    return [
        # one small patch of crossing fibers: the least work a fit can be, bound by latency and launches
        _case("step", (8, 8, 8), name="step_patch", patch=8),
        # a sweep of 16 small volumes with a noise level each, Rician likelihood
        _case("step", (10, 10, 10), name="step_sweep", vols=16, loss="nll", patch=10),
        # crossing-fiber benchmark layout: one b = 0 and an odd count, two fibers, no neighbour priors
        _case("step", (17, 20, 10), name="step_crossing", n_meas=193, b0=1, K=2),
        # tractography-phantom shape: 40^3, strong weighting, five fibers, Rician likelihood, coherence priors
        _case("step", (40, 40, 40), name="step_disco", n_meas=364, b0=4, shells=4, bmax=13192.0, snr=50.0, K=5,
              loss="nll", spatial=True, iters=8),
        # bundle phantom: full nuisance calibration with the Rician likelihood
        _case("step", (64, 64, 64), name="step_bundle", n_meas=360, b0=20, bmax=4000.0, snr=20.0, loss="nll",
              cal=True, spatial=True, iters=4),
        # a batch of unlike volumes (sizes, odd measurement counts, measurements in acquisition order)
        _case("step", (56, 61, 47), name="step_batch", vols=4, unlike=True, mask="ellipsoid", n_meas=271, b0=13,
              mixed=True, spatial=True, conn=26, iters=4),
        # the whole brain, 740,110 voxels x 288 measurements: the benchmark's workload
        _case("step", (145, 174, 145), name="step_brain", mask="brain", n_meas=288, b0=18, spatial=True, iters=4),
        # a program's own optimiser on a small patch
        _case("grad", (12, 11, 9), name="grad_patch", n_meas=97, b0=7, mixed=True),
        # the same with calibration and the Rician likelihood on a phantom
        _case("grad", (40, 40, 40), name="grad_bundle", n_meas=360, b0=20, bmax=4000.0, snr=20.0, loss="nll",
              cal=True, spatial=True),
        # and on a brain at half resolution
        _case("grad", (97, 116, 97), name="grad_brain", mask="ellipsoid", n_meas=288, b0=18, spatial=True),
        # a host framework that owns device memory evaluates a block of voxels
        _case("noalloc", (61, 53, 47), name="noalloc_block", n_meas=288, b0=18, mixed=True),
        # quality control of a stored whole-volume fit on its data
        _case("review", (73, 87, 73), name="review_slabs", mask="ellipsoid", n_meas=288, b0=18, spatial=True),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "grad", "grad", "noalloc", "review"])
    lo, hi = {"step": (300, 500_000), "grad": (300, 300_000), "noalloc": (200, 400_000), "review": (2000, 250_000)}[kind]
    voxels = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    edge = voxels ** (1 / 3)
    nx, ny = (max(3, round(edge * rng.uniform(0.75, 1.3))) for _ in range(2))
    nz = max(3, round(voxels / (nx * ny)))
    K = rng.choice([1, 2, 3, 3, 3, 4, 5])
    shells = rng.choice([1, 2, 3, 3, 4])
    n_meas = round(math.exp(rng.uniform(math.log(33), math.log(400))))
    n_meas = min(n_meas, max(33, int(7e8 / (voxels * K))))   # no more than the whole brain's work
    b0 = max(1, min(n_meas // 4, rng.choice([1, n_meas // 18, n_meas // 16])))
    loss = rng.choice(["mse", "mse", "nll"]) if kind in ("step", "grad") else "mse"
    cal = kind in ("step", "grad") and rng.random() < 0.3
    vols = rng.choice([1, 1, 1, 3, 6]) if kind == "step" and voxels < 60_000 else 1
    if vols > 1:
        nx, ny, nz = (max(3, round(n / vols ** (1 / 3))) for n in (nx, ny, nz))
    return _case(kind, (nx, ny, nz), vols=vols, unlike=vols > 1 and rng.random() < 0.5,
                 mask=rng.choice(["full", "ellipsoid"]) if min(nx, ny, nz) >= 6 else "full", n_meas=n_meas, b0=b0,
                 shells=shells, bmax=float(rng.choice([1500, 3000, 4000, 8000])), mixed=rng.random() < 0.5,
                 snr=float(rng.choice([10, 20, 30, 50])), K=K, loss=loss, cal=cal,
                 spatial=kind != "noalloc" and rng.random() < 0.6, conn=rng.choice([6, 6, 26]),
                 patch=rng.choice([8, 16, 16, 20]), iters=16 if voxels < 30_000 else 4)


# -- inputs --------------------------------------------------------------------------------------
def _parts(case):
    """(shape, measurements) of each volume; in an unlike batch the later ones are smaller and shorter."""
    out = []
    for i in range(case["vols"]):
        s = 1.0 - 0.13 * i if case["unlike"] else 1.0
        n = case["n_meas"] - (37 * i if case["unlike"] else 0)
        out.append((tuple(max(3, round(case[a] * s)) for a in ("nx", "ny", "nz")), max(case["b0"] + 12, n)))
    return out


def _mask(shape, kind):
    if kind == "full":
        return np.ones(shape, np.uint8)
    semi = (52.8, 63.4, 52.8) if kind == "brain" else tuple(n / 2 for n in shape)
    ax = [((np.arange(n) - (n - 1) / 2) / a) ** 2 for n, a in zip(shape, semi)]
    return (ax[0][:, None, None] + ax[1][None, :, None] + ax[2][None, None, :] <= 1.0).astype(np.uint8)


def _scheme(case, n_meas):
    """b-values and unit b-vectors: b = 0 first and shell after shell, or mixed as acquired."""
    b0, S = case["b0"], case["shells"]
    per = [(n_meas - b0) // S + (1 if i >= S - (n_meas - b0) % S else 0) for i in range(S)]
    bvals, bvecs = [np.zeros(b0)], [np.zeros((b0, 3))]
    for i, n in enumerate(per):
        t = np.arange(n) + 0.5
        z, phi = 1.0 - t / n, math.pi * (1 + 5 ** 0.5) * t + i
        r = np.sqrt(1 - z * z)
        bvals.append(np.full(n, round(case["bmax"] * (i + 1) / S)))
        bvecs.append(np.stack([r * np.cos(phi), r * np.sin(phi), z], 1))
    bvals, bvecs = np.concatenate(bvals), np.concatenate(bvecs)
    if case["mixed"]:
        order = np.random.RandomState(n_meas).permutation(n_meas)
        bvals, bvecs = bvals[order], bvecs[order]
    return bvals.astype(np.float32), bvecs.astype(np.float32)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda")


def _anatomy(case, shape, mask, g):
    """Smooth truth of one volume: fractions [V, K + 3], directions [V, K, 3], f_intra [V]."""
    K = case["K"]
    xyz = torch.nonzero(torch.as_tensor(mask, device="cuda")).float()
    xyz = xyz / max(shape)
    wave = 4.0 + 4.0 * _rand(g, 3, 4 * K + 4)
    field = torch.sin(xyz @ wave + 6.28 * _rand(g, 4 * K + 4)) + 0.15 * _randn(g, xyz.shape[0], 4 * K + 4)
    logits = 0.8 * field[:, :K + 3]
    logits[:, 2] += 1.2          # a main fiber, a second one, weaker others
    if K > 1:
        logits[:, 3] += 0.6
    dirs = field[:, K + 3:4 * K + 3].reshape(-1, K, 3) + 0.3 * _randn(g, 1, K, 3)
    dirs = dirs / dirs.norm(dim=2, keepdim=True).clamp_min(1e-3)
    fin = 0.5 + 0.1 * field[:, 4 * K + 3].clamp(-1, 1)
    return torch.log_softmax(logits, 1), dirs, fin


def _signal(case, truth, bvals, bvecs, g):
    """Raw magnitudes [V, N] (S0 near 1000) of a stick-and-zeppelin tissue with its own diffusivities."""
    logf, dirs, fin = truth
    f = logf.exp()
    V, K = f.shape[0], case["K"]
    b = torch.as_tensor(bvals, device="cuda")
    gv = torch.as_tensor(bvecs, device="cuda")
    out = torch.empty((V, len(bvals)), device="cuda")
    par, perp = 1.5e-3 + 0.5e-3 * _rand(g, V, 1), 0.3e-3 + 0.3e-3 * _rand(g, V, 1)
    amp, s0, sd = 1.0, 900.0 + 200.0 * _rand(g, V, 1), 1.0 / case["snr"]
    if case["cal"]:
        amp = torch.exp(0.02 * _randn(g, 1, len(bvals)))
        s0 = s0 * (1.0 + 0.15 * torch.sin(torch.linspace(0, 5, V, device="cuda"))[:, None])
    for i in range(0, V, 1 << 16):
        c = slice(i, min(V, i + (1 << 16)))
        s = sum(f[c, j, None] * torch.exp(-b * d) for j, d in ((0, D_CSF), (1, D_GM), (K + 2, D_RES)))
        for k in range(K):
            x = (dirs[c, k] @ gv.T) ** 2
            e = fin[c, None] * torch.exp(-b * par[c] * x)
            s += f[c, 2 + k, None] * (e + (1 - fin[c, None]) * torch.exp(-b * (par[c] * x + perp[c] * (1 - x))))
        s = s * amp
        out[c] = s0[c] * torch.hypot(s + sd * _randn(g, *s.shape), sd * _randn(g, *s.shape))
    return out


def _theta(case, truth, g):
    """Raw parameters of a fit part of the way to the truth."""
    logf, dirs, fin = truth
    V, K = logf.shape[0], case["K"]
    th = torch.empty((V, 4 * K + 5), device="cuda")
    th[:, 0] = 0.54 + 0.05 * _randn(g, V)
    th[:, 1:K + 4] = logf + 1.8 + 0.15 * _randn(g, V, K + 3)
    th[:, K + 4:4 * K + 4] = (dirs * (1.0 + 0.2 * _rand(g, V, K, 1)) + 0.08 * _randn(g, V, K, 3)).reshape(V, 3 * K)
    th[:, 4 * K + 4] = torch.logit(fin) + 0.2 * _randn(g, V)
    return th


def _groups(case, parts, g):
    """Packed group parameters: sigma_log, alpha, beta and b_lr of every volume."""
    out = []
    for _, n in parts:
        n4 = (n + 3) // 4 * 4
        p = torch.zeros(4 + 2 * n4 + 512, device="cuda")
        p[0] = math.log(1.1 / case["snr"])
        if case["cal"]:
            p[4:4 + n] = 0.02 * _randn(g, n)
            p[4 + n4:4 + n4 + n] = 0.003 * _randn(g, n)
            p[4 + 2 * n4:] = 0.1 * _randn(g, 512)
        out.append(p)
    return torch.cat(out)


def _moments(case, parts, V, g):
    """Adam moments of a fit under way, on the scale of its gradients: m, v of the voxel parameters
    [V, 4K + 5] and of the packed group parameters."""
    Q = 4 * case["K"] + 5
    n = case["n_meas"]
    s = 0.2 * n / V if case["loss"] == "mse" else 0.1 * n * case["snr"]
    v = (s * (0.5 + _rand(g, V, Q))) ** 2
    m = 0.3 * v.sqrt() * _randn(g, V, Q)
    gp = sum(4 + 2 * ((k + 3) // 4 * 4) + 512 for _, k in parts)
    sg = (1.0 if case["loss"] == "mse" else V * case["snr"]) * (0.5 + _rand(g, gp))
    return m, v, 0.1 * sg * _randn(g, gp), sg ** 2


def _options(case, **kw):
    pri = dict(lam_rep=0.01, lam_sparse=0.02)
    if case["spatial"]:
        pri.update(lam_sp=0.01, lam_dir=0.005, connectivity=case["conn"])
    return prism.options(K=case["K"], loss=case["loss"], calibration=case["cal"], patch_dim=case["patch"], **pri, **kw)


def _make(case, seed):
    """The inputs of a case: volumes (with their truth left out), theta, groups and the generator."""
    g = torch.Generator("cuda").manual_seed(seed)
    parts, vols, thetas = _parts(case), [], []
    for shape, n in parts:
        mask = _mask(shape, case["mask"])
        bvals, bvecs = _scheme(case, n)
        truth = _anatomy(case, shape, mask, g)
        vols.append(Volume(mask, _signal(case, truth, bvals, bvecs, g), bvals, bvecs))
        thetas.append(_theta(case, truth, g))
    return parts, vols, torch.cat(thetas), _groups(case, parts, g), g


def prepare(case, seed):
    parts, vols, theta, groups, g = _make(case, seed)
    V, kind = theta.shape[0], case["kind"]
    st = dict(case=case, theta=theta, groups=groups)
    if kind == "step":
        f = prism.Fitter(vols, _options(case))
        blob = bytearray(f.state())
        struct.pack_into("<i", blob, 20, STEP0)
        m, v, gm, gv = _moments(case, parts, V, g)
        at = len(blob) - 12 * (theta.numel() + groups.numel())
        for x in (theta, m, v, groups, gm, gv):
            raw = x.cpu().numpy().tobytes()
            blob[at:at + len(raw)] = raw
            at += len(raw)
        f.load_state(bytes(blob))
        st["fitter"] = f
    elif kind == "grad":
        st["fitter"] = prism.Fitter(vols, _options(case))
        theta.requires_grad_(True)
        groups.requires_grad_(True)
    elif kind == "noalloc":
        st.update(signal=vols[0].signal, bvals=vols[0].bvals, bvecs=vols[0].bvecs, lib=_lib.load(), opts=_options(case),
                  grad=torch.empty_like(theta), loss=torch.empty(1, dtype=torch.float64, device="cuda"))
    else:
        vols[0].init = theta
        K = case["K"]
        st.update(volume=vols[0], opts=_options(case),
                  maps=tuple(torch.empty(s, device="cuda") for s in ((V,), (V, K + 3), (V,), (V, K, 3))))
    return st


# The objective is a double sum of terms computed in 32 bits; a program keeps it as the 32-bit
# number that it is good for, which is what run() returns.
def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "step":
        f = st["fitter"]
        f.step(case["iters"])
        return {"theta": f.params(), "groups": f.groups_device()}
    if kind == "grad":
        loss = prism.PrismLoss.apply(st["theta"], st["groups"], st["fitter"])
        gth, ggr = torch.autograd.grad(loss, [st["theta"], st["groups"]])
        return {"loss": loss.detach().float(), "g_theta": gth, "g_groups": ggr}
    if kind == "noalloc":
        o, p = st["opts"], lambda t: ctypes.c_void_p(t.data_ptr())   # noqa: E731
        V, N = st["signal"].shape
        _lib.check(st["lib"].prism_grad_noalloc(
            p(st["signal"]), st["bvals"].ctypes.data, st["bvecs"].ctypes.data, p(st["theta"]), V, N, case["K"],
            o.lam_rep, o.lam_sparse, o.tau, p(st["grad"]), p(st["loss"]),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)))
        return {"loss": st["loss"].float(), "g_theta": st["grad"]}
    with prism.Fitter(st["volume"], st["opts"], slabs=_slabs(case)) as f:
        loss, yhat = f.forward(want_yhat=True)
        s0, fr, fin, dirs = f.stitch(out=st["maps"])
    return {"loss": loss.float(), "yhat": yhat, "s0": s0, "fractions": fr, "f_intra": fin, "dirs": dirs}


def _slabs(case):
    """30-slice slabs with a 5-slice overlap; thinner ones for a volume of few slices."""
    return (30, 5) if case["nz"] > 30 else (max(2, case["nz"] // 2), 1)


def work(case):
    parts = _parts(case)
    vox = [int(np.count_nonzero(_mask(s, case["mask"]))) for s, _ in parts]
    K, Q, kind = case["K"], 4 * case["K"] + 5, case["kind"]
    it = case["iters"] if kind == "step" else 1
    # flops of a (voxel, measurement) pair, multiply-add = 2: model and adjoint, 26 per fiber and 4;
    # Rician terms 70, calibration 11; a review evaluates the model alone, about half of it
    per = 4 + 26 * K + (70 if case["loss"] == "nll" else 0) + (11 if case["cal"] else 0)
    flops = sum(v * n for v, (_, n) in zip(vox, parts)) * per * it * (0.5 if kind == "review" else 1)
    sig = sum(4 * v * n for v, (_, n) in zip(vox, parts))
    V = sum(vox)
    if kind == "step":   # the signal once; parameters and moments read, written and read out
        return {"bytes": sig + V * Q * 4 * 7, "flops": flops}
    if kind == "review":  # the signal in, the predicted signal and the maps out
        return {"bytes": 2 * sig + V * Q * 8, "flops": flops}
    return {"bytes": sig + V * Q * 8, "flops": flops}


# -- the same in 64 bits, from the model's equations -----------------------------------------------
def _neighbours(mask, patch, conn):
    """Neighbour voxels in the same patch, [E, V] (V where there is none), and forward face pairs in the mask."""
    m = torch.as_tensor(mask, device="cuda").bool()
    idx = torch.full([n + 2 for n in m.shape], -1, dtype=torch.long, device="cuda")
    V = int(m.sum())
    xyz = torch.nonzero(m)
    x, y, z = (xyz + 1).T
    idx[x, y, z] = torch.arange(V, device="cuda")
    offs = [(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1) if (i, j, k) != (0, 0, 0)]
    rows, pairs = [], []
    for o in offs:
        n = idx[x + o[0], y + o[1], z + o[2]]
        if sum(map(abs, o)) == 1 and sum(o) == 1:
            pairs.append((torch.nonzero(n >= 0)[:, 0], n[n >= 0]))
        if conn == 6 and sum(map(abs, o)) != 1:
            continue
        same = (n >= 0) & (torch.div(xyz + torch.tensor(o, device="cuda"), patch, rounding_mode="floor")
                           == torch.div(xyz, patch, rounding_mode="floor")).all(1)
        rows.append(torch.where(same, n, V))
    return torch.stack(rows), pairs, xyz


def _upsample(blr, xyz, shape):
    """Trilinear values of the 8^3 grid at the voxels, cell centres aligned to the volume."""
    U = 0.0
    lo, w = [], []
    for a in range(3):
        u = ((xyz[:, a].double() + 0.5) * 8 / shape[a] - 0.5).clamp(0, 7)
        i = u.floor().clamp(max=6)
        lo.append(i.long())
        w.append(u - i)
    for cx in (0, 1):
        for cy in (0, 1):
            for cz in (0, 1):
                wt = 1.0
                for a, c in enumerate((cx, cy, cz)):
                    wt = wt * (w[a] if c else 1 - w[a])
                U = U + wt * blr[lo[0] + cx, lo[1] + cy, lo[2] + cz]
    return U


def _split(theta, K):
    S0 = torch.nn.functional.softplus(theta[:, 0])
    f = torch.softmax(theta[:, 1:K + 4], 1)
    v = theta[:, K + 4:4 * K + 4].reshape(-1, K, 3)
    return S0, f, v / v.norm(dim=2, keepdim=True).clamp_min(1e-12), torch.sigmoid(theta[:, 4 * K + 4])


class _Exact:
    """Objective of one volume in 64 bits, its gradient by automatic differentiation."""

    def __init__(self, case, vol, patch_volume=None):
        self.case, self.vol = case, vol
        self.b = torch.as_tensor(vol.bvals, device="cuda").double()
        self.g = torch.as_tensor(vol.bvecs, device="cuda").double()
        self.y = vol.signal.double()
        self.y = self.y / self.y[:, self.b <= B0_MAX].mean(1, keepdim=True)
        self.nbr, self.pairs, self.xyz = _neighbours(vol.mask, case["patch"], case["conn"])
        self.count = (self.nbr < self.y.shape[0]).sum(0).double()

    def predict(self, theta, gp, U, rows):
        K = self.case["K"]
        S0, f, d, fin = _split(theta, K)
        s = f[:, 0, None] * torch.exp(-self.b * D_CSF) + f[:, 1, None] * torch.exp(-self.b * D_GM)
        s = s + f[:, K + 2, None] * torch.exp(-self.b * D_RES)
        for k in range(K):
            x = (d[:, k] @ self.g.T) ** 2
            e = fin[:, None] * torch.exp(-self.b * D_PAR * x)
            s = s + f[:, 2 + k, None] * (e + (1 - fin[:, None]) * torch.exp(-self.b * (D_PAR * x + D_PERP * (1 - x))))
        s = S0[:, None] * s
        if self.case["cal"]:
            n = len(self.b)
            n4 = (n + 3) // 4 * 4
            s = torch.exp(gp[4:4 + n]) * torch.exp(U[rows])[:, None] * s + gp[4 + n4:4 + n4 + n]
        return s

    def value_and_grad(self, theta, gp, want_grad=True):
        """J and dJ/dtheta, dJ/dgroups (64 bits)."""
        case, K, V, N = self.case, self.case["K"], theta.shape[0], len(self.b)
        theta, gp = theta.detach().requires_grad_(True), gp.detach().requires_grad_(True)
        n4, inv = (N + 3) // 4 * 4, 1.0 / V
        total = torch.zeros((), dtype=torch.float64, device="cuda")
        U = _upsample(gp[4 + 2 * n4:].reshape(8, 8, 8), self.xyz, self.vol.mask.shape) if case["cal"] else None
        Ud = U.detach().requires_grad_(True) if case["cal"] else None
        step = max(1, int(1.2e7 / N))
        for i in range(0, V, step):      # data term, a block of voxels at a time
            rows = slice(i, min(V, i + step))
            yh, y = self.predict(theta[rows], gp, Ud, rows), self.y[rows]
            if case["loss"] == "mse":
                J = (yh - y).square().sum() * inv
            else:
                s2, a = torch.exp(2 * gp[0]), yh.abs()
                J = (2 * gp[0] + (y - a) ** 2 / (2 * s2) - torch.log(torch.special.i0e(y * a / s2))).sum()
            if want_grad:
                J.backward()
            total += J.detach()
        S0, f, d, _ = _split(theta, K)
        J = torch.zeros((), dtype=torch.float64, device="cuda")
        w = f[:, 2:2 + K]
        for i in range(K):
            for j in range(i):
                J = J + 0.01 * inv * (w[:, i] * w[:, j] * (d[:, i] * d[:, j]).sum(1).abs()).sum()
        # the gate compares 32-bit values, as the method's threshold does
        J = J + 0.02 * inv * (w * (w.detach() < float(np.float32(0.15)))).sum()
        if case["spatial"]:
            has, cnt = self.count > 0, self.count.clamp_min(1)
            fp = torch.cat([f, f.new_zeros(1, K + 3)])
            u = f - sum(fp[r] for r in self.nbr) / cnt[:, None]
            a = u.abs()
            rho = torch.where(a <= 0.05, 0.5 * u * u, 0.05 * (a - 0.025))
            J = J + 0.01 * inv * rho[has].sum()
            dp = torch.cat([d, d.new_zeros(1, K, 3)])
            for r in self.nbr:
                ok = (r < V).double()
                J = J + 0.005 * inv * ((1 - (d * dp[r]).sum(2) ** 2).sum(1) * ok / cnt).sum()
        if case["cal"]:
            J = J + 1e-3 * (gp[4:4 + N].square().mean() + gp[4 + n4:4 + n4 + N].square().mean()
                            + gp[4 + 2 * n4:].square().mean())
            B = torch.exp(Ud)
            for p, q in self.pairs:
                J = J + 1e-3 * inv * torch.sqrt((B[q] - B[p]) ** 2 + 1e-6).sum()
        total += J.detach()
        if want_grad:
            J.backward()
            if case["cal"]:
                U.backward(Ud.grad)
            if case["loss"] == "mse":
                gp.grad = gp.grad if gp.grad is not None else torch.zeros_like(gp)
                gp.grad[0] = 0.0
        return total, theta.grad, gp.grad


def _adam(x, grad, m, v, t):
    m.mul_(0.9).add_(grad, alpha=1 - 0.9)
    v.mul_(0.999).addcmul_(grad, grad, value=1 - 0.999)
    x -= 1e-2 / (1 - 0.9 ** t) * m / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)


def exact(case, seed):
    parts, vols, theta, groups, g = _make(case, seed)
    V = theta.shape[0]
    K, kind = case["K"], case["kind"]
    cost = sum(len(v.bvals) * v.signal.shape[0] for v in vols) * (case["iters"] if kind == "step" else 1)
    if cost * (K + (3 if case["loss"] == "nll" else 1)) > 4.5e9:
        return None
    th, gp = theta.double(), groups.double()
    vo = np.cumsum([0] + [v.signal.shape[0] for v in vols])
    go = np.cumsum([0] + [4 + 2 * ((n + 3) // 4 * 4) + 512 for _, n in parts])
    if kind == "review":
        return _exact_review(case, vols[0], th, gp)
    models = [_Exact(case, v) for v in vols]
    m, v, gm, gv = (x.double() for x in _moments(case, parts, V, g)) if kind == "step" else (None,) * 4
    for it in range(case["iters"] if kind == "step" else 1):
        J, gth, ggp = [], torch.zeros_like(th), torch.zeros_like(gp)
        for i, mod in enumerate(models):
            a, b = slice(vo[i], vo[i + 1]), slice(go[i], go[i + 1])
            j, gth[a], ggp[b] = mod.value_and_grad(th[a], gp[b])
            J.append(j)
        if kind != "step":
            out = {"loss": sum(J), "g_theta": gth, "g_groups": ggp}
            if kind == "noalloc":
                out.pop("g_groups")
                out["loss"] = out["loss"].reshape(1)
            return out
        _adam(th, gth, m, v, STEP0 + it + 1)
        train = torch.zeros_like(gp)      # sigma with the Rician likelihood, the rest with calibration
        for i, (_, n) in enumerate(parts):
            train[go[i]] = case["loss"] == "nll"
            n4 = (n + 3) // 4 * 4
            for at, k in ((4, n), (4 + n4, n), (4 + 2 * n4, 512)):
                train[go[i] + at:go[i] + at + k] = case["cal"]
        new = gp.clone()
        _adam(new, ggp, gm, gv, STEP0 + it + 1)
        gp = torch.where(train > 0, new, gp)
    return {"theta": th, "groups": gp}


def _exact_review(case, vol, th, gp):
    K, (slab, lap) = case["K"], _slabs(case)
    nz = vol.mask.shape[2]
    z = torch.nonzero(torch.as_tensor(vol.mask, device="cuda"))[:, 2]
    J, yhat, z0 = [], [], 0
    while True:
        z1 = min(z0 + slab, nz)
        rows = torch.nonzero((z >= z0) & (z < z1))[:, 0]
        if len(rows):
            part = Volume(np.ascontiguousarray(vol.mask[:, :, z0:z1]), vol.signal[rows], vol.bvals, vol.bvecs)
            mod = _Exact(case, part)
            with torch.no_grad():
                J.append(mod.value_and_grad(th[rows], gp, False)[0])
                yhat.append(mod.predict(th[rows], gp, None, None))
        if z1 >= nz:
            break
        z0 += slab - lap
    # a stored fit is one set of parameters, so overlapping slabs blend equal estimates
    S0, f, d, fin = _split(th, K)
    return {"loss": torch.stack(J), "yhat": torch.cat([y.reshape(-1) for y in yhat]), "s0": S0, "fractions": f,
            "f_intra": fin, "dirs": d}
