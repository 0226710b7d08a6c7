"""Performance cases: what a user of the reconstruction library has it do, through the
public Python entry points (`Reconstructor`, `BatchReconstructor`, `DeviceInference`).

A case names a `kind` (which calls one pass makes) and its sizes:

  apply     Toeplitz applies (A*A + lam) x of one or several vectors
  solve     a fixed number of CG iterations on a loaded kernel and right-hand side
  separate  firm_kernel + firm_backproject: K-hat and A*b
  fused     both spreading channels in one call: K-hat and A*b
  whole     fused sums, learned preconditioner, a few PCG iterations: a reconstruction
  forward   the forward projector A V on every image's half disc
  residual  the data term |b - A V|^2
  batch     several reconstructions of uneven size as one unit

Inputs are made on the GPU from the seed alone: Gaussian-blob phantoms, analytic
projections with shifts and white noise, views that are Haar-uniform, mixed (von
Mises-Fisher about three axes), a polar cap, or a conical tilt series.
"""
import math

import numpy as np
import torch

from paper_1307_5824_gb300 import BatchReconstructor, Reconstructor
from paper_1307_5824_gb300 import _lib as L
from paper_1307_5824_gb300.learned import DeviceInference

DEV = "cuda:0"
LAM = 1e-3                      # relative Tikhonov weight of every workload with a CTF


def listed():
    return [
        # one operator apply of a small volume: the launch latency of an iteration
        dict(name="apply_n32", kind="apply", N=32, vectors=1),
        # plain CG at the middle size, as a caller that loaded summed shards runs it
        dict(name="cg_n64", kind="solve", N=64, precond=False, iters=10),
        # preconditioned CG at the largest volume: the loop of a full-size reconstruction
        dict(name="pcg_n128", kind="solve", N=128, precond=True, iters=5),
        # the smallest reconstruction's sums: 200 views, no CTF, few points per brick
        dict(name="sums_n32_m200", kind="separate", N=32, M=200, W=6, bf16=False, views="haar", groups=0),
        # the ordinary size: uneven views, shifts, four defocus groups, FP32 images
        dict(name="sums_n64_m5000", kind="separate", N=64, M=5000, W=6, bf16=False, views="mixed", groups=4),
        # a tilt series at the paper's size, no CTF, the wider default window
        dict(name="sums_n96_m10000_w7", kind="separate", N=96, M=10000, W=7, bf16=False, views="rct", groups=0),
        # strongly uneven views (85% within 15 degrees of a pole), pose channel separate
        dict(name="sums_n128_m40000_cap", kind="separate", N=128, M=40000, W=6, bf16=True, views="cap", groups=8),
        # the headline size: 50,000 BF16 images, both channels in one call
        dict(name="fused_n128_m50000", kind="fused", N=128, M=50000, W=6, bf16=True, views="haar", groups=20),
        # a whole reconstruction of a modest image set with the learned preconditioner
        dict(name="whole_n96_m2500", kind="whole", N=96, M=2500, W=6, bf16=False, views="mixed", groups=3, iters=4),
        # projections of a volume at the ordinary size (residual maps, refinement)
        dict(name="forward_n64_m5000", kind="forward", N=64, M=5000, W=6, bf16=False, views="mixed", groups=4),
        # the data term of the L-curve at the largest volume
        dict(name="residual_n128_m15000", kind="residual", N=128, M=15000, W=6, bf16=True, views="haar", groups=20),
        # many uneven reconstructions as one captured unit
        dict(name="batch_16", kind="batch", n=16, m_lo=1000, m_hi=8000, W=6, iters=6),
    ]


# the number of images at most, by volume edge (what users run at that size, and no
# drawn case costs more than the largest listed one)
M_MOST = {32: 4000, 48: 8000, 64: 12000, 80: 12000, 96: 15000, 128: 40000}


def draw(rng):
    kind = rng.choice(["apply", "solve", "separate", "separate", "fused", "whole", "forward", "residual", "batch"])
    N = rng.choice([32, 48, 64, 80, 96, 128])
    if kind == "apply":
        return dict(kind=kind, N=N, vectors=rng.randint(1, 24))
    if kind == "solve":
        pre = rng.random() < 0.5
        return dict(kind=kind, N=N, precond=pre, iters=rng.randint(2, 5) if pre else rng.randint(4, 10))
    if kind == "batch":
        lo = rng.randint(300, 2000)
        return dict(kind=kind, n=rng.randint(2, 12), m_lo=lo, m_hi=lo + rng.randint(1, 5000), W=6, iters=rng.randint(2, 6))
    top = M_MOST[N] if kind not in ("forward", "residual") else M_MOST[N] // 2
    M = int(round(math.exp(rng.uniform(math.log(100), math.log(top)))))
    case = dict(kind=kind, N=N, M=M, W=rng.choice([6, 6, 6, 7]), bf16=rng.random() < 0.5,
                views=rng.choice(["haar", "mixed", "cap", "rct"]), groups=rng.choice([0, 1, 4, 8, 20]))
    if kind == "whole":
        case["iters"] = rng.randint(2, 4)
    return case


# ------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------
def _frame(d, psi):
    """Rotations whose third row is the direction d, with in-plane angle psi."""
    a = np.where(np.abs(d[:, 2:3]) < 0.9, np.array([[0.0, 0.0, 1.0]]), np.array([[1.0, 0.0, 0.0]]))
    e1 = np.cross(a, d)
    e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
    e2 = np.cross(d, e1)
    c, s = np.cos(psi)[:, None], np.sin(psi)[:, None]
    return np.stack([c * e1 + s * e2, c * e2 - s * e1, d], axis=1)


def _polar(w, phi):
    s = np.sqrt(np.maximum(0.0, 1.0 - w * w))
    return np.stack([s * np.cos(phi), s * np.sin(phi), w], axis=1)


def _views(kind, M, rng):
    """(M, 3, 3) rotations of a view distribution."""
    def haar(n):
        d = rng.standard_normal((n, 3))
        return d / np.linalg.norm(d, axis=1, keepdims=True)

    if kind == "haar":
        d = haar(M)
    elif kind == "rct":                                        # 60 degree tilt series
        d = _polar(np.full(M, 0.5), rng.uniform(0, 2 * np.pi, M))
    elif kind == "cap":                                        # 85% within 15 degrees of z
        n = int(0.85 * M)
        d = np.concatenate([_polar(rng.uniform(np.cos(np.pi / 12), 1.0, n), rng.uniform(0, 2 * np.pi, n)), haar(M - n)])
    else:                                                      # 70% von Mises-Fisher, 30% Haar
        n = int(0.7 * M)
        w = 1.0 + np.log(rng.uniform(1e-12, 1.0, n) * (1 - np.exp(-40.0)) + np.exp(-40.0)) / 20.0
        loc = _polar(w, rng.uniform(0, 2 * np.pi, n))
        axes = _frame(haar(3), np.zeros(3))
        d = np.concatenate([np.einsum("mi,mij->mj", loc, axes[rng.integers(0, 3, n)]), haar(M - n)])
    d = d[rng.permutation(M)]
    return _frame(d, rng.uniform(0, 2 * np.pi, M))


def _groups(n):
    """Defocus groups from 1.0 to 3.5 um, 300 kV, Cs 2 mm, 2.8 A pixels."""
    t = np.zeros((n, 6))
    t[:, 0] = np.linspace(1.0, 3.5, n) * 1e4 if n > 1 else 2e4
    t[:, 1], t[:, 2], t[:, 3], t[:, 4] = 300.0, 2.0, 0.07, 2.8
    return t


def _blobs(N, rng, n=40):
    d = rng.standard_normal((n, 3))
    d *= (0.3 * N * rng.uniform(0, 1, n) ** (1 / 3) / np.linalg.norm(d, axis=1))[:, None]
    return d, rng.uniform(1.5, 4.0, n), rng.uniform(0.5, 1.0, n)


def _volume(blobs, N):
    x = torch.arange(N, device=DEV, dtype=torch.float64) - N // 2
    c, s, a = (torch.from_numpy(v).to(DEV) for v in blobs)
    g = [torch.exp(-(x[None] - c[:, k:k + 1]) ** 2 / (2 * s[:, None] ** 2)) for k in range(3)]
    return torch.einsum("bz,by,bx->zyx", g[2] * a[:, None], g[1], g[0]).float().contiguous()


def _images(blobs, R, shifts, N, bf16, gen, snr=0.1):
    """Analytic projections of the blobs plus white noise, (M, N, N) on the GPU."""
    M = R.shape[0]
    out = torch.empty((M, N, N), device=DEV, dtype=torch.bfloat16 if bf16 else torch.float32)
    x = torch.arange(N, device=DEV, dtype=torch.float32) - N // 2
    c, s, a = (torch.from_numpy(v).to(DEV) for v in blobs)
    pref = (a * s * math.sqrt(2 * math.pi)).float()
    s2 = (2 * s * s).float()
    sigma = None
    for i in range(0, M, 4096):
        P = (torch.einsum("mij,bj->mbi", R[i:i + 4096, :2], c) + shifts[i:i + 4096, None]).float()
        gx = torch.exp(-(x - P[:, :, 0:1]) ** 2 / s2[None, :, None])
        gy = torch.exp(-(x - P[:, :, 1:2]) ** 2 / s2[None, :, None]) * pref[None, :, None]
        im = torch.matmul(gy.transpose(1, 2), gx)
        if sigma is None:
            sigma = (im.var() / snr).sqrt()
        out[i:i + 4096] = im + sigma * torch.randn(im.shape, device=DEV, generator=gen)
    return out


def _problem(N, M, views, groups, bf16, seed, images=True):
    """Poses, shifts, group ids, images and phantom of one reconstruction."""
    rng = np.random.default_rng([seed, N, M])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rng.integers(1 << 40)))
    blobs = _blobs(N, rng)
    R = torch.from_numpy(_views(views, M, rng)).to(DEV)
    shifts = torch.from_numpy(rng.uniform(-2, 2, (M, 2))).to(DEV)
    gid = torch.from_numpy(rng.integers(0, max(groups, 1), M).astype(np.int32)).to(DEV)
    p = dict(N=N, M=M, R=R.reshape(M, 9).contiguous(), shifts=shifts, gid=gid, groups=_groups(groups), blobs=blobs)
    if images:
        p["images"] = _images(blobs, R, shifts, N, bf16, gen)
    return p


def _model_sums(N, seed):
    """A Ker half box and right-hand side such as summed image shards give: a spectrum
    that falls as 1 / |k| inside the ball, modulated by a CTF and by uneven views, and
    the operator's image of a phantom plus noise."""
    rng = np.random.default_rng([seed, N])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(rng.integers(1 << 40)))
    f = torch.fft.fftfreq(2 * N, device=DEV, dtype=torch.float64) * 2 * N
    k3, k2, k1 = torch.meshgrid(f, f, f, indexing="ij")
    r = (k1 * k1 + k2 * k2 + k3 * k3).sqrt()
    a = torch.from_numpy(_frame(rng.standard_normal((1, 3)), np.zeros(1))[0, 2]).to(DEV)
    a = a / a.norm()
    cosine = (k1 * a[0] + k2 * a[1] + k3 * a[2]) / r.clamp(min=1.0)
    dens = 1e4 / r.clamp(min=1.0) * (0.2 + torch.sin(0.3 + 40 * (r / (2 * N)) ** 2) ** 2) * (1.2 - cosine ** 2)
    noise = torch.rand(r.shape, device=DEV, generator=gen, dtype=torch.float64)
    noise = noise + torch.flip(torch.roll(noise, (-1, -1, -1), (0, 1, 2)), (0, 1, 2))
    dens = torch.where(r <= N, dens * (0.5 + 0.5 * noise), torch.zeros_like(r))
    ker = torch.fft.fftshift(torch.fft.ifftn(dens).real) * (2.0 * N) ** 3
    half = torch.cat([ker[:, :, N:], ker[:, :, :1]], dim=2).float().contiguous()
    V = _volume(_blobs(N, rng), N).double()
    rhs = _apply64(_khat64(half), V, 0.0)
    rhs = (rhs + 0.3 * rhs.std() * torch.randn(rhs.shape, device=DEV, generator=gen, dtype=torch.float64)).float()
    return half, rhs.contiguous(), V.float().contiguous()


def _vectors(V, n):
    """n volumes as a block method has them: the phantom turned and scaled."""
    turned = [torch.rot90(V, j % 4, (1 + j // 4 % 2, 0)) * (1.0 + 0.1 * j) for j in range(n)]
    return torch.stack(turned).contiguous()


class _State(dict):
    """What a program holds between passes; its plan goes with it."""


def prepare(case, seed):
    kind = case["kind"]
    s = _State(case=case)
    if kind in ("apply", "solve"):
        N = case["N"]
        half, rhs, V = _model_sums(N, seed)
        rec = Reconstructor(N, 0, lam=LAM, device=DEV)
        rec.load_sums(half, rhs)
        s.update(rec=rec, x=V, y=torch.empty_like(V), half=half, rhs=rhs)
        if kind == "apply":
            s.update(x=_vectors(V, case["vectors"]))
            s.update(y=torch.empty_like(s["x"]))
        elif case["precond"]:
            rec.set_precond(L.FIRM_PRECOND_CIRCULANT)
        return s
    if kind == "batch":
        recs, items = [], []
        for j, (N, M, views, groups) in enumerate(_batch_list(case)):
            p = _problem(N, M, views, groups, False, seed * 64 + j)
            recs.append(Reconstructor(N, M, groups=p["groups"], W=case["W"], lam=LAM, device=DEV))
            items.append(dict(M=M, R=p["R"], images=p["images"], shifts=p["shifts"], group=p["gid"],
                              x=torch.empty((N, N, N), device=DEV)))
        bat = BatchReconstructor(recs, device=DEV)
        bat.set_items(items)
        s.update(bat=bat, out=[it["x"] for it in items])
        return s
    N, M = case["N"], case["M"]
    p = _problem(N, M, case["views"], case["groups"], case["bf16"], seed, images=kind != "forward")
    rec = Reconstructor(N, M, groups=p["groups"], W=case["W"], lam=LAM, device=DEV, fused=kind in ("fused", "whole"),
                        img_dtype=L.FIRM_IMG_BF16 if case["bf16"] else L.FIRM_IMG_F32)
    s.update(p, rec=rec)
    if kind in ("forward", "residual"):
        s["V"] = _volume(p["blobs"], N)
        if kind == "forward":
            s["out"] = torch.empty((M, (L.disc_size(N) + 1) // 2, 2), device=DEV)
    else:
        s["khat"] = torch.empty(rec.half_shape(), device=DEV)
        s["rhs"] = torch.empty((N, N, N), device=DEV)
    if kind == "whole":
        s["x"] = torch.empty((N, N, N), device=DEV)
        s["net"] = DeviceInference(_network(seed))
    return s


def _batch_list(case):
    """(N, M, views, groups) of every reconstruction of a batch (its shape, not its data)."""
    rng = np.random.default_rng([case["n"], case["m_lo"], case["m_hi"]])
    return [(int(rng.choice([48, 64, 80, 96])), int(rng.integers(case["m_lo"], case["m_hi"] + 1)), "mixed",
             int(rng.integers(1, 5))) for _ in range(case["n"])]


def _network(seed):
    """Weights of a trained network's size whose output follows the shells' usual trend
    (a multiplier that grows with the radius), in the parameter layout of the library."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed * 7 + 3)
    w, parts = (1024, 256, 256, 1024), []
    for i in range(3):
        scale = math.sqrt(2.0 / w[i]) * (0.03 if i == 2 else 1.0)
        parts.append(torch.randn(w[i + 1] * w[i], device=DEV, generator=gen) * scale)
        parts.append(torch.zeros(w[i + 1], device=DEV))
    parts[5] = torch.log(1.0 + torch.arange(1024, device=DEV) // 16).float()
    return torch.cat(parts)


# ------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------
def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "apply":
        for j in range(case["vectors"]):
            s["rec"].toeplitz_apply(s["x"][j], s["y"][j])
        return s["y"]
    if kind == "solve":
        s["rec"].cg_solve(s["y"], case["iters"])
        return s["y"]
    if kind == "batch":
        s["bat"].run(case["iters"])
        s["bat"].wait()
        return s["out"]
    rec = s["rec"]
    if kind == "separate":
        rec.kernel(s["R"], s["gid"], khat_out=s["khat"])
        rec.backproject(s["images"], s["shifts"], s["R"], s["gid"], rhs_out=s["rhs"])
        return {"khat": s["khat"], "rhs": s["rhs"]}
    if kind == "fused":
        rec.kernel_backproject(s["images"], s["shifts"], s["R"], s["gid"], khat_out=s["khat"], rhs_out=s["rhs"])
        return {"khat": s["khat"], "rhs": s["rhs"]}
    if kind == "whole":
        rec.kernel_backproject(s["images"], s["shifts"], s["R"], s["gid"], khat_out=s["khat"], rhs_out=s["rhs"])
        s["net"].apply(rec)
        rec.cg_solve(s["x"], case["iters"])
        return {"khat": s["khat"], "rhs": s["rhs"], "table": s["net"].y, "x": s["x"]}
    if kind == "forward":
        return rec.forward(s["V"], s["R"], s["gid"], out=s["out"])
    a, b = rec.data_residual(s["V"], s["images"], s["shifts"], s["R"], s["gid"])
    return np.array([a, b])


# ------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------
def _fft_flops(L):
    return 2.5 * L ** 3 * math.log2(L ** 3)                   # a real transform of L^3 points


def _iter_work(N, precond):
    b = 4.0 * (2 * N * 2 * N * (N + 1)) + 8.0 * N ** 3        # K-hat, one vector in, one out
    f = 2 * _fft_flops(2 * N)
    if precond:
        b += 4.0 * N * N * (N // 2 + 1) + 8.0 * N ** 3
        f += 2 * _fft_flops(N)
    return b, f


def _sums_work(N, M, W, esz, kernel=True, rhs=True):
    nH = (L.disc_size(N) + 1) / 2
    b, f = M * (72.0 + 4.0), 0.0
    if kernel:
        b += 4.0 * (2 * N * 2 * N * (N + 1))
        f += M * nH * W ** 3 * 2 + _fft_flops(4 * N) + _fft_flops(2 * N)
    if rhs:
        b += M * (16.0 + N * N * esz) + 4.0 * N ** 3
        f += M * nH * W ** 3 * 4 + M * 2.5 * N * N * math.log2(N * N) + 2 * _fft_flops(2 * N)
    return b, f


def work(case):
    kind = case["kind"]
    if kind == "apply":
        b, f = (case["vectors"] * v for v in _iter_work(case["N"], False))
    elif kind == "solve":
        b, f = (case["iters"] * v for v in _iter_work(case["N"], case["precond"]))
    elif kind == "batch":
        b = f = 0.0
        for N, M, _, _ in _batch_list(case):
            sb, sf = _sums_work(N, M, case["W"], 4)
            ib, if_ = _iter_work(N, False)
            b, f = b + sb + case["iters"] * ib, f + sf + case["iters"] * if_
    else:
        N, M, W, esz = case["N"], case["M"], case["W"], 2 if case["bf16"] else 4
        nH = (L.disc_size(N) + 1) / 2
        if kind == "forward":
            b = 4.0 * N ** 3 + M * (76.0 + 8.0 * nH)
            f = M * nH * W ** 3 * 4 + 2 * _fft_flops(2 * N)
        elif kind == "residual":
            b = 4.0 * N ** 3 + M * (92.0 + N * N * esz)
            f = M * nH * W ** 3 * 4 + 2 * _fft_flops(2 * N) + M * 2.5 * N * N * math.log2(N * N)
        else:
            b, f = _sums_work(N, M, W, esz)
            if kind == "whole":
                ib, if_ = _iter_work(N, True)
                b, f = b + case["iters"] * ib, f + case["iters"] * if_
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------------
# The same results in 64 bits, with torch alone
# ------------------------------------------------------------------------------------
def _khat64(half):
    """Circulant spectrum (real, (2N)^3) of the Ker half box [n3+N][n2+N][n1]."""
    N = half.shape[0] // 2
    c = torch.zeros((2 * N,) * 3, dtype=torch.float64, device=half.device)
    h = half.double()
    i = torch.arange(2 * N, device=half.device)
    keep = i[i != N]
    lag = torch.where(keep < N, keep, keep - 2 * N)
    pos = lag >= 0
    a = keep[pos]
    c[keep[:, None, None], keep[None, :, None], a[None, None, :]] = \
        h[(lag + N)[:, None, None], (lag + N)[None, :, None], lag[pos][None, None, :]]
    b, lb = keep[~pos], lag[~pos]
    c[keep[:, None, None], keep[None, :, None], b[None, None, :]] = \
        h[(N - lag)[:, None, None], (N - lag)[None, :, None], (-lb)[None, None, :]]
    return torch.fft.fftn(c).real


def _apply64(khat, V, lam):
    N = V.shape[0]
    y = torch.fft.ifftn(khat * torch.fft.fftn(V.double(), s=(2 * N,) * 3)).real
    return y[:N, :N, :N] + lam * V


def _chan64(half):
    """T. Chan's optimal circulant spectrum on the N^3 grid."""
    N = half.shape[0] // 2
    c = torch.fft.ifftn(_khat64(half)).real                   # the circulant column
    i = torch.arange(N, device=c.device)
    out = torch.zeros((N,) * 3, dtype=torch.float64, device=c.device)
    parts = [(i, (N - i) / N), ((i + N) % (2 * N), i / N)]    # lags i and i - N
    for z, wz in parts:
        for y, wy in parts:
            for x, wx in parts:
                out += c[z][:, y][:, :, x] * (wz[:, None, None] * wy[None, :, None] * wx[None, None, :])
    return torch.fft.fftn(out).real


def _solve64(half, rhs, iters, precond):
    N = rhs.shape[0]
    khat, lam = _khat64(half), LAM * float(half[N, N, 0])
    b = rhs.double()
    d = 1.0 / (_chan64(half).clamp(min=0.0) + lam) if precond else None
    P = (lambda r: torch.fft.ifftn(d * torch.fft.fftn(r)).real) if precond else (lambda r: r)
    x, r = torch.zeros_like(b), b.clone()
    z = P(r)
    p, rz = z.clone(), (r * z).sum()
    for _ in range(iters):
        q = _apply64(khat, p, lam)
        a = rz / (p * q).sum()
        x, r = x + a * p, r - a * q
        z = P(r)
        new = (r * z).sum()
        p, rz = z + new / rz * p, new
    return x


_TAPS = 10


def _window(t):
    beta = 2.3 * _TAPS
    u = 1.0 - (2.0 * t / _TAPS) ** 2
    return torch.where(u > 0, torch.exp(beta * (u.clamp(min=0.0).sqrt() - 1.0)), torch.zeros_like(t))


def _window_ft(u):
    """Fourier transform of the window at the frequencies u (cycles per cell)."""
    x, w = np.polynomial.legendre.leggauss(400)
    t = torch.from_numpy(x * _TAPS / 2).to(DEV)
    phi = _window(t) * torch.from_numpy(w * _TAPS / 2).to(DEV)
    return (torch.cos(2 * math.pi * u[:, None] * t[None]) * phi[None]).sum(1)


def _half_disc(N):
    h = N // 2
    k = [(0, b) for b in range(h + 1)]
    k += [(a, b) for a in range(1, h + 1) for b in range(-h, h + 1) if a * a + b * b <= h * h]
    return torch.tensor(k, device=DEV, dtype=torch.float64)


def _ctf64(N, groups, gid, K):
    if groups.shape[0] == 0:
        return torch.ones((gid.shape[0], K.shape[0]), dtype=torch.float64, device=DEV)
    out = []
    r = K.norm(dim=1)
    for df, kv, cs, amp, pix, bf in groups:
        U = kv * 1e3
        lam = 6.62607015e-34 / math.sqrt(2 * 9.1093837015e-31 * 1.602176634e-19 * U *
                                         (1 + 1.602176634e-19 * U / (2 * 9.1093837015e-31 * 299792458.0 ** 2))) * 1e10
        q = (r / (N * pix)) ** 2
        chi = math.pi * lam * df * q - 0.5 * math.pi * cs * 1e7 * lam ** 3 * q * q
        out.append(-torch.sin(chi + amp) * torch.exp(-bf * q / 4))
    return torch.stack(out)[gid.long()]


class _Grid:
    """Nonuniform points of the slices on a grid of 2 L cells per axis."""

    def __init__(self, R, K, N, modes):
        self.L, self.G = modes, 2 * modes
        y = torch.einsum("ka,maj->mkj", K / N, R.reshape(-1, 3, 3)[:, :2]).reshape(-1, 3) * self.G
        i0 = torch.ceil(y - _TAPS / 2)
        self.w = [torch.stack([_window(i0[:, a] + l - y[:, a]) for l in range(_TAPS)]) for a in range(3)]
        self.i0 = [i0[:, a].long() for a in range(3)]
        n = torch.arange(-(modes // 2), modes - modes // 2, device=DEV)
        self.n, self.dec = n % self.G, 1.0 / _window_ft(n.double() / self.G)

    def taps(self):
        G = self.G
        for a in range(_TAPS):
            iz, wz = (self.i0[2] + a) % G, self.w[2][a]
            for b in range(_TAPS):
                iy, wy = (iz * G + (self.i0[1] + b) % G) * G, wz * self.w[1][b]
                for c in range(_TAPS):
                    yield iy + (self.i0[0] + c) % G, wy * self.w[0][c]

    def scale(self):
        d = self.dec
        return d[:, None, None] * d[None, :, None] * d[None, None, :]

    def crop(self, f):
        return f[self.n][:, self.n][:, :, self.n]

    def type1(self, wts):
        """2 Re sum_p wts_p exp(+i <n, xi_p>) on the centred modes."""
        cols = torch.view_as_real(wts) if wts.is_complex() else wts[:, None]
        g = torch.zeros((self.G ** 3, cols.shape[1]), dtype=torch.float64, device=DEV)
        for idx, w in self.taps():
            g.index_add_(0, idx, cols * w[:, None])
        g = torch.view_as_complex(g) if wts.is_complex() else g[:, 0]
        f = torch.fft.ifftn(g.reshape((self.G,) * 3).to(torch.complex128)).real * float(self.G) ** 3
        return 2 * self.crop(f) * self.scale()

    def type2(self, V):
        """sum_n V_n exp(-i <n, xi_p>) at every point."""
        pad = torch.zeros((self.G,) * 3, dtype=torch.float64, device=DEV)
        ix = self.n
        pad[ix[:, None, None], ix[None, :, None], ix[None, None, :]] = V.double() * self.scale()
        f = torch.view_as_real(torch.fft.fftn(pad)).reshape(-1, 2)
        out = torch.zeros((self.i0[0].shape[0], 2), dtype=torch.float64, device=DEV)
        for idx, w in self.taps():
            out += f[idx] * w[:, None]
        return torch.view_as_complex(out)


def _image_dft64(images, shifts, K, N):
    kx, ky = (K[:, 0] % N).long(), (K[:, 1] % N).long()
    out = torch.empty((images.shape[0], K.shape[0]), dtype=torch.complex128, device=DEV)
    for i in range(0, images.shape[0], 1024):
        im = torch.fft.ifftshift(images[i:i + 1024].double(), dim=(1, 2))
        ph = 2 * math.pi / N * (shifts[i:i + 1024] @ K.T)
        out[i:i + 1024] = torch.fft.fft2(im)[:, ky, kx] * torch.polar(torch.ones_like(ph), ph)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("apply", "solve"):
        N = case["N"]
        half, rhs, V = _model_sums(N, seed)
        if kind == "apply":
            khat, lam = _khat64(half), LAM * float(half[N, N, 0])
            return torch.stack([_apply64(khat, x, lam) for x in _vectors(V, case["vectors"])])
        return _solve64(half, rhs, case["iters"], case["precond"])
    if kind == "batch":
        return None
    N, M = case["N"], case["M"]
    K = _half_disc(N)
    if M * K.shape[0] > 2.2e7:                                # the sums take too long in 64 bits
        return None
    p = _problem(N, M, case["views"], case["groups"], case["bf16"], seed, images=kind != "forward")
    h = _ctf64(N, p["groups"], p["gid"], K)
    if kind in ("forward", "residual"):
        grid = _Grid(p["R"], K, N, N)
        A = grid.type2(_volume(p["blobs"], N)).reshape(M, -1) * h
        if kind == "forward":
            return torch.view_as_real(A)
        b = _image_dft64(p["images"], p["shifts"], K, N)
        c = torch.full((K.shape[0],), 2.0, dtype=torch.float64, device=DEV)
        c[0] = 1.0
        return np.array([float((c * (b - A).abs() ** 2).sum()), float((c * b.abs() ** 2).sum())])
    once = torch.ones(K.shape[0], dtype=torch.float64, device=DEV)
    once[0] = 0.5                                             # k = 0 is its own mirror image
    ker = _Grid(p["R"], K, N, 2 * N).type1((h * h * once).reshape(-1))
    half = torch.cat([ker[:, :, N:], ker[:, :, :1]], dim=2)
    khat = _khat64(half)[:, :, :N + 1].contiguous()
    g = (_image_dft64(p["images"], p["shifts"], K, N) * h * once).reshape(-1)
    out = {"khat": khat, "rhs": _Grid(p["R"], K, N, N).type1(g)}
    if kind == "whole":
        out.update(table=None, x=None)
    return out
