"""The calls whose speed this repository keeps track of, through the public entry points.

Seven kinds of call stand for what a program does with the library:

  gradient  one gradient of the objective (tmbir_gradient) at a start image
  recon     one run of the fast gradient method (tmbir_reconstruct) from the FBP start
  setup     R*g and the FBP start of a new sinogram on a geometry the context already holds
  newscan   the same for a scan with its own angles: context, workspace, kernel, R*g, FBP start
  refine    the learned refiner applied to a batch of start images
  train     the refiner's forward and backward pass of a training batch, gradients out
  upsample  the Lanczos-3 transfer of a volume to the next level

`groups` lists the geometry groups of a context as side:slices:angles, joined by "+".
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2603_28756_gb300 as tm

PRIOR = dict(p=1.2, q=2.0, c=0.01, sigma=0.1, lam=1.0)
LIMITED = 2 * math.pi / 3
DEV = "cuda"
L2_BYTES = 100e6  # iterates below this can stay on the chip from one iteration to the next


def listed():
    return [
        # one gradient of a single small slice, as a program with a solver of its own asks for it:
        # launches and host work
        dict(name="gradient-1x64sq-45ang", kind="gradient", groups="64:1:45", span=math.pi),
        # the plain method on one slice: a preview, or a first look at a parameter
        dict(name="recon-1x128sq-90ang-50it", kind="recon", groups="128:1:90", span=math.pi, iters=50, bf16=False,
             nonneg=False),
        # the coarsest level of the hierarchical form: BF16 spectra
        dict(name="recon-64x512sq-128ang-bf16", kind="recon", groups="512:64:128", span=LIMITED, iters=2, bf16=True,
             nonneg=False),
        # the batched workload
        dict(name="recon-64x1024sq-256ang-10it", kind="recon", groups="1024:64:256", span=math.pi, iters=10,
             bf16=False, nonneg=False),
        # the finest level of the hierarchical form, limited angle
        dict(name="recon-32x2048sq-128ang-10it", kind="recon", groups="2048:32:128", span=LIMITED, iters=10,
             bf16=False, nonneg=False),
        # an uneven batch: sides, slice counts and angle counts mixed in one context
        dict(name="recon-uneven-4sides-5it", kind="recon",
             groups="512:7:180+1024:5:64+1024:3:181+1536:4:128+2048:3:90", span=math.pi, iters=5, bf16=False,
             nonneg=True),
        # the detector width of the nano-CT data
        dict(name="recon-6x2560sq-150ang-5it", kind="recon", groups="2560:6:150", span=math.pi, iters=5, bf16=False,
             nonneg=False),
        # the next slab of a scan: a new sinogram on a geometry that is already built
        dict(name="setup-16x2048sq-128ang", kind="setup", groups="2048:16:128", span=LIMITED),
        # the first slab of a scan with its own angles
        dict(name="newscan-4x512sq-181ang", kind="newscan", groups="512:4:181", span=math.pi),
        # the learned warm start of a batch of slices
        dict(name="refine-8x1024sq", kind="refine", H=1024, W=1024, batch=8),
        # one batch of the refiner's training
        dict(name="train-8x1024sq", kind="train", H=1024, W=1024, batch=8),
        # the step from one level of the hierarchy to the next
        dict(name="upsample-32x1024sq", kind="upsample", N=1024, S=32),
    ]


SIDES = (64, 128, 256, 512, 1024, 1536, 2048, 2560)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _slices(rng, N, voxels):
    return _log(rng, 1, max(1, min(128, voxels // (N * N))))


def draw(rng):
    kind = rng.choice(["gradient", "recon", "recon", "recon", "setup", "newscan", "refine", "train", "upsample"])
    span = rng.choice([math.pi, math.pi, LIMITED])
    if kind == "gradient":
        N = rng.choice(SIDES)
        return dict(kind=kind, groups="%d:%d:%d" % (N, _slices(rng, N, 1 << 24), _log(rng, 30, 256)), span=span)
    if kind == "recon":
        if rng.random() < 0.25:  # uneven
            gs = ["%d:%d:%d" % (N, _slices(rng, N, 1 << 23), _log(rng, 30, 200))
                  for N in sorted(rng.choice(SIDES) for _ in range(rng.randint(2, 5)))]
            return dict(kind=kind, groups="+".join(gs), span=span, iters=rng.randint(2, 8), bf16=False,
                        nonneg=rng.random() < 0.5)
        if rng.random() < 0.25:  # a coarse level
            N = rng.choice((256, 512))
            return dict(kind=kind, groups="%d:%d:%d" % (N, _slices(rng, N, 1 << 24), _log(rng, 30, 256)), span=span,
                        iters=2, bf16=True, nonneg=False)
        N = rng.choice(SIDES)
        return dict(kind=kind, groups="%d:%d:%d" % (N, _slices(rng, N, 1 << 26), _log(rng, 30, 256)), span=span,
                    iters=rng.randint(3, 12), bf16=False, nonneg=rng.random() < 0.25)
    if kind == "setup":
        N = rng.choice(SIDES)
        return dict(kind=kind, groups="%d:%d:%d" % (N, _slices(rng, N, 1 << 25), _log(rng, 30, 200)), span=span)
    if kind == "newscan":
        N = rng.choice((64, 128, 256, 512, 1024))
        return dict(kind=kind, groups="%d:%d:%d" % (N, _slices(rng, N, 1 << 20), _log(rng, 30, 200)), span=span)
    if kind == "upsample":
        N = rng.choice((64, 128, 256, 512, 768, 1024, 1280))
        return dict(kind=kind, N=N, S=_slices(rng, N, 1 << 25))
    H, W = _log(rng, 64, 1400), _log(rng, 64, 1400)  # refine, train: images need not be square
    return dict(kind=kind, H=H, W=W, batch=_log(rng, 1, max(1, min(8, (1 << 23) // (H * W)))))


# ---------------------------------------------------------------- inputs
def _groups(case):
    return [tuple(int(v) for v in g.split(":")) for g in case["groups"].split("+")]


def _theta(na, span):
    return np.arange(na, dtype=np.float64) * (span / na)


def _ellipsoids(seed, N, S, n=20):
    """Centres in the disc of radius 0.55 N/2, semi-axes U[0.05, 0.35] N/2 shrunk to stay inside 0.95 N/2, z
    semi-axes U[0.1, 0.5] S, densities U[0, 1] (rows x0, y0, a, b, phi, rho, z0, cz)."""
    r = np.random.default_rng(seed)
    R = N / 2.0
    rad, ang = 0.55 * R * np.sqrt(r.uniform(0, 1, n)), r.uniform(0, 2 * np.pi, n)
    a, b = r.uniform(0.05, 0.35, n) * R, r.uniform(0.05, 0.35, n) * R
    s = np.minimum(1.0, (0.95 * R - rad) / np.maximum(a, b))
    cz = np.maximum(r.uniform(0.1, 0.5, n) * S, 0.6)
    return np.stack([rad * np.cos(ang), rad * np.sin(ang), a * s, b * s, r.uniform(0, np.pi, n), r.uniform(0, 1, n),
                     r.uniform(0, S, n), cz], 1)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) + 500)


def _sinogram(seed, N, S, theta):
    """Exact line integrals of the ellipsoids at the bin centres, with Gaussian noise of 1 % of the maximum."""
    th = torch.tensor(theta, device=DEV)[None, :, None]
    s = (torch.arange(N, device=DEV, dtype=torch.float64) - N / 2.0)[None, None, :]
    z = (torch.arange(S, device=DEV, dtype=torch.float64) + 0.5)[:, None, None]
    g = torch.zeros(S, len(theta), N, device=DEV, dtype=torch.float64)
    for x0, y0, a, b, phi, rho, z0, cz in _ellipsoids(seed, N, S):
        f2 = torch.clamp(1 - ((z - z0) / cz) ** 2, min=0)
        al2 = (a * torch.cos(th - phi)) ** 2 + (b * torch.sin(th - phi)) ** 2
        sp = s - (x0 * torch.cos(th) + y0 * torch.sin(th))
        g += 2 * rho * a * b * torch.sqrt(torch.clamp(al2 * f2 - sp * sp, min=0)) / al2 * torch.sqrt(f2)
    return (g + 0.01 * float(g.max()) * torch.randn(g.shape, device=DEV, dtype=torch.float64,
                                                    generator=_gen(seed))).float()


def _sinograms(case, seed):
    return torch.cat([_sinogram(seed * 64 + i, N, S, _theta(na, case["span"])).reshape(-1)
                      for i, (N, S, na) in enumerate(_groups(case))])


def _images(seed, H, W, S):
    """Sections of the ellipsoids (H x W windows of the phantom's side) with noise, and the same without."""
    N = max(H, W)
    y = (torch.arange(H, device=DEV, dtype=torch.float32) - H / 2)[None, :, None]
    x = (torch.arange(W, device=DEV, dtype=torch.float32) - W / 2)[None, None, :]
    z = (torch.arange(S, device=DEV, dtype=torch.float32) + 0.5)[:, None, None]
    v = torch.zeros(S, H, W, device=DEV)
    for x0, y0, a, b, phi, rho, z0, cz in _ellipsoids(seed, N, S):
        u = (x - x0) * math.cos(phi) + (y - y0) * math.sin(phi)
        w = -(x - x0) * math.sin(phi) + (y - y0) * math.cos(phi)
        v += rho * ((u / a) ** 2 + (w / b) ** 2 + ((z - z0) / cz) ** 2 <= 1)
    return v + 0.1 * torch.randn(v.shape, device=DEV, generator=_gen(seed)), v


def _context(case):
    return tm.Context([tm.Group(N=N, angles=list(_theta(na, case["span"])), n_slices=S, span=case["span"])
                       for N, S, na in _groups(case)])


def _training_batch(case, seed):
    """A batch as the training step hands it to the network: images over their RMS, and the gradient of the mean
    squared error of a network that is still near zero."""
    x, t = _images(seed, case["H"], case["W"], case["batch"])
    s = x.double().square().mean((1, 2), keepdim=True).sqrt().float()
    return x / s, -2 * ((t - x) / s) / x.numel()


LAYERS = ((1, 32), (32, 32), (32, 32), (32, 1))


def _params():
    """The refiner's weights: He-normal, the last layer a tenth of that, small biases."""
    r = np.random.default_rng(7)
    p = []
    for ci, co in LAYERS:
        gain = math.sqrt(2 / (9 * ci)) * (0.1 if co == 1 else 1)
        p += [r.normal(0, gain, 9 * ci * co), r.normal(0, 0.02, co)]
    return np.concatenate(p).astype(np.float32)


def _net(case):
    net = tm.CNN(case["H"], case["W"], max_batch=case["batch"])
    net.set_weights(_params())
    return net


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("gradient", "recon", "setup"):
        st["sino"] = _sinograms(case, seed)
        st["ctx"] = ctx = _context(case)
        st["atg"], st["x0"] = ctx.build_operator_fbp(st["sino"])
        if kind == "gradient":
            st["prm"] = tm.Params(**PRIOR)
        if kind == "recon":
            st["x"] = torch.empty_like(st["x0"])
            st["prm"] = tm.Params(**PRIOR, max_iter=case["iters"], bf16=case["bf16"], nonneg=case["nonneg"])
    elif kind == "newscan":
        st["sino"] = _sinograms(case, seed)
    elif kind == "refine":
        st["net"] = _net(case)
        st["x"] = _images(seed, case["H"], case["W"], case["batch"])[0].reshape(-1)
    elif kind == "train":
        st["net"] = _net(case)
        st["x"], st["gout"] = (t.reshape(-1) for t in _training_batch(case, seed))
    else:
        st["ctx"] = tm.Context([tm.Group(N=64, angles=[0.0], n_slices=1)])
        st["x"] = _images(seed, case["N"], case["N"], case["S"])[0].reshape(-1)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "gradient":
        return st["ctx"].gradient(st["x0"], st["atg"], st["prm"])
    if kind == "recon":
        st["x"].copy_(st["x0"])
        st["ctx"].reconstruct(st["x"], st["atg"], st["prm"])
        return st["x"]
    if kind == "setup":
        return st["ctx"].build_operator_fbp(st["sino"], st["atg"], st["x0"])
    if kind == "newscan":
        return _context(case).build_operator_fbp(st["sino"])
    if kind == "refine":
        return st["net"].apply(st["x"], case["batch"])
    if kind == "train":
        return st["net"].net_backward(st["x"], st["gout"], case["batch"])
    return st["ctx"].upsample_lanczos3(st["x"], case["S"], case["N"])


# ---------------------------------------------------------------- what a pass cannot do without
def _gradient_flops(N, S):
    """Real row transforms of length 2N and complex column transforms of length 2N, both ways, and the 13 neighbour
    pairs of each voxel."""
    M, lg = 2 * N, math.log2(2 * N)
    return S * (2 * N * 2.5 * M * lg + 2 * (N + 1) * 5 * M * lg + 13 * 15 * N * N)


def work(case):
    kind = case["kind"]
    if kind in ("gradient", "recon", "setup", "newscan"):
        gs = _groups(case)
        vox = sum(S * N * N for N, S, na in gs)
        sino = sum(S * na * N for N, S, na in gs)
        if kind == "gradient":
            return {"bytes": 12 * vox, "flops": sum(_gradient_flops(N, S) for N, S, na in gs)}
        if kind == "recon":
            # x_k, x_{k-1} and R*g in, x_{k+1} out, every iteration once the iterates outgrow the L2
            its = case["iters"]
            return {"bytes": 16 * vox * its if 16 * vox > L2_BYTES else 12 * vox,
                    "flops": its * sum(_gradient_flops(N, S) for N, S, na in gs)}
        # two back-projections: radial transforms, and the 2D transform that leads to N x N pixels
        fl = sum(2 * S * (na * 5 * N * math.log2(N) + 2 * 2.5 * N * N * math.log2(N * N)) for N, S, na in gs)
        if kind == "newscan":  # and the kernel's transform
            fl += sum(5 * 4 * N * N * math.log2(4 * N * N) for N, S, na in gs)
        return {"bytes": 4 * sino + 8 * vox, "flops": fl}
    if kind == "upsample":
        n = case["S"] * case["N"] ** 2
        return {"bytes": 4 * n + 16 * n, "flops": 11 * (n + 2 * n)}
    px = case["batch"] * case["H"] * case["W"]
    macs = 2 * 9 * 32 + 2 * 9 * 32 * 32
    if kind == "refine":
        return {"bytes": 8 * px, "flops": 2 * macs * px}
    return {"bytes": 12 * px, "flops": 6 * macs * px}


# ---------------------------------------------------------------- the same in 64 bits
def _kernel(N, theta):
    """K(d) = (1/N) sum_a D(e_a . d) on |dx|, |dy| < N, D(t) = sum over |k| <= N/2 - 1 of cos(2 pi k t / N)."""
    d = torch.arange(-(N - 1), N, device=DEV, dtype=torch.float64)
    K = torch.zeros(2 * N - 1, 2 * N - 1, device=DEV, dtype=torch.float64)
    for th in theta:
        t = d[:, None] * math.sin(th) + d[None, :] * math.cos(th)
        e = (t - N * torch.round(t / N)) * (math.pi / N)
        den = torch.sin(e)
        D = torch.sin((N - 1) * e) / den
        K += torch.where(den == 0, float(N - 1), D)
    return K / N


def _spectrum(N, theta):
    K = _kernel(N, theta)
    C = torch.zeros(2 * N, 2 * N, device=DEV, dtype=torch.float64)
    i = torch.arange(-(N - 1), N, device=DEV) % (2 * N)
    C[i[:, None], i[None, :]] = K
    return torch.fft.rfft2(C).real.contiguous()


def _apply(x, spec):
    N = x.shape[-1]
    out = torch.empty_like(x)
    for z in range(0, x.shape[0], 4):
        f = torch.fft.rfft2(x[z:z + 4], s=(2 * N, 2 * N)) * spec
        out[z:z + 4] = torch.fft.irfft2(f, s=(2 * N, 2 * N))[:, :N, :N]
    return out


def _adjoint(g, N, theta):
    """R* g = sum_a p_a(e_a . x), p_a the trigonometric polynomial of period N through the projection without its
    Nyquist term: a grid 16 times finer by FFT, then 12-point Lagrange interpolation (error about 1e-12)."""
    S = g.shape[0]
    over, taps = 16, 12
    c = torch.arange(N, device=DEV, dtype=torch.float64) - N // 2
    out = torch.zeros(S, N, N, device=DEV, dtype=torch.float64)
    step = max(1, int(2 ** 27 // (S * N)))
    for a, th in enumerate(theta):
        G = torch.fft.rfft(torch.roll(g[:, a], -(N // 2), 1))
        G[:, N // 2] = 0
        P = over * torch.fft.irfft(G, n=over * N)
        for r in range(0, N, step):
            t = (c[r:r + step, None] * math.sin(th) + c[None, :] * math.cos(th)) * over
            i0 = torch.floor(t)
            u = t - i0
            i0 = i0.long() - (taps // 2 - 1)
            for j in range(taps):
                w = torch.ones_like(u)
                for m in range(taps):
                    if m != j:
                        w = w * ((u + (taps // 2 - 1) - m) / (j - m))
                out[:, r:r + step] += w * P[:, (i0 + j) % (over * N)]
    return out


def _ramp(g):
    """Linear convolution of every projection with the unit-pitch Ram-Lak kernel."""
    N = g.shape[-1]
    n = torch.arange(-N, N, device=DEV, dtype=torch.float64)
    h = torch.where(n % 2 != 0, -1.0 / (math.pi * n) ** 2, 0.0)
    h[N] = 0.25
    M = 4 * N
    f = torch.fft.irfft(torch.fft.rfft(g, M) * torch.fft.rfft(h, M), M)
    return f[..., N:2 * N]


def _prior(y, pr):
    """Gradient of the qGGMRF prior over the 26-neighbourhood, each pair once."""
    total = 6 + 12 / math.sqrt(2) + 8 / math.sqrt(3)
    G = torch.zeros_like(y)
    S, N = y.shape[0], y.shape[1]
    for dz in (0, 1):
        for dy in (-1, 0, 1):
            for dx in (-1, 0, 1):
                if (dz, dy, dx) <= (0, 0, 0):
                    continue
                w = 1 / math.sqrt(dz + dy * dy + dx * dx) / total
                ys, yd = slice(max(0, -dy), N - max(0, dy)), slice(max(0, dy), N + min(0, dy))
                xs, xd = slice(max(0, -dx), N - max(0, dx)), slice(max(0, dx), N + min(0, dx))
                for z in range(0, S - dz, 8):
                    e = min(S - dz, z + 8)
                    d = y[z:e, ys, xs] - y[z + dz:e + dz, yd, xd]
                    r = 1 / (1 + (d.abs() / (pr["c"] * pr["sigma"])) ** (pr["q"] - pr["p"]))
                    f = (w / pr["sigma"] ** 2) * d * r * (pr["p"] + (pr["q"] - pr["p"]) * r)
                    G[z:e, ys, xs] += f
                    G[z + dz:e + dz, yd, xd] -= f
    return G


def _lambda_max(N, spec):
    v = torch.full((1, N, N), 1.0 / N, device=DEV, dtype=torch.float64)
    lam = 0.0
    for _ in range(100):
        w = _apply(v, spec)
        lam = float((v * w).sum())
        v = w / w.norm()
    return lam


def _group_exact(case, g, N, theta):
    """(R*g, FBP start) of one group."""
    return _adjoint(g, N, theta), _adjoint(_ramp(g), N, theta) * (case["span"] / len(theta))


def _iterations(x, atg, spec, L, iters, nonneg):
    xp, t, beta = x, 1.0, 0.0
    for _ in range(iters):
        y = x + beta * (x - xp)
        G = _apply(y, spec) - atg + PRIOR["lam"] * _prior(y, PRIOR)
        xn = y - G / L
        if nonneg:
            xn = xn.clamp(min=0)
        if float((G * (xn - x)).sum()) > 0:
            t = 1.0
        else:
            t = 0.5 * (1 + math.sqrt(1 + 4 * t * t))
        beta = (t - 1) / (0.5 * (1 + math.sqrt(1 + 4 * t * t)))
        x, xp = xn, x
    return x


def _conv_net(x, p):
    """1 -> 32 -> 32 -> 32 -> 1, 3x3, zero padding, ReLU after the first three layers."""
    at = 0
    h = x[:, None]
    for layer, (ci, co) in enumerate(LAYERS):
        w = p[at:at + 9 * ci * co].reshape(co, ci, 3, 3)
        at += 9 * ci * co
        b = p[at:at + co]
        at += co
        h = F.conv2d(h, w, b, padding=1)
        if layer < 3:
            h = torch.relu(h)
    return h[:, 0]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("refine", "train"):
        p = torch.tensor(_params().astype(np.float64), device=DEV, requires_grad=kind == "train")
        if kind == "refine":
            x = _images(seed, case["H"], case["W"], case["batch"])[0].double()
            out = torch.empty_like(x)
            with torch.no_grad():
                for b in range(x.shape[0]):
                    s = x[b].square().mean().sqrt()
                    out[b] = x[b] + s * _conv_net(x[b:b + 1] / s, p)[0]
            return out.reshape(-1)
        x, gout = (t.double() for t in _training_batch(case, seed))
        gins = []
        for b in range(x.shape[0]):
            xb = x[b:b + 1].clone().requires_grad_(True)
            (_conv_net(xb, p) * gout[b:b + 1]).sum().backward()
            gins.append(xb.grad.reshape(-1))
        return p.grad, torch.cat(gins)
    if kind == "upsample":
        S, N = case["S"], case["N"]
        x = _images(seed, N, N, S)[0].double()
        o = torch.tensor([2.5, 1.5, 0.5, -0.5, -1.5, -2.5], dtype=torch.float64)
        w = torch.sinc(o) * torch.sinc(o / 3)
        w = (w / w.sum()).tolist()

        def up(v, dim):
            v = v.movedim(dim, -1)
            pad = F.pad(v, (2, 3))
            odd = sum(w[t] * pad[..., t:t + v.shape[-1]] for t in range(6))
            return torch.stack([v, odd], -1).flatten(-2).movedim(-1, dim)

        return up(up(x, 2), 1).reshape(-1)
    sino = _sinograms(case, seed).double()
    at, outs = 0, []
    for N, S, na in _groups(case):
        theta = _theta(na, case["span"])
        g = sino[at:at + S * na * N].reshape(S, na, N)
        at += S * na * N
        atg, x0 = _group_exact(case, g, N, theta)
        if kind in ("setup", "newscan"):
            outs.append((atg, x0))
            continue
        spec = _spectrum(N, theta)
        if kind == "gradient":
            outs.append((_apply(x0, spec) - atg + PRIOR["lam"] * _prior(x0, PRIOR),))
            continue
        L = 1.01 * _lambda_max(N, spec) + PRIOR["lam"] * 2 * 2 / PRIOR["sigma"] ** 2
        outs.append((_iterations(x0, atg, spec, L, case["iters"], case["nonneg"]),))
    cat = tuple(torch.cat([o[j].reshape(-1) for o in outs]) for j in range(len(outs[0])))
    return cat if len(cat) > 1 else cat[0]
