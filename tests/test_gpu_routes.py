"""Kernels and dispatch rules at the sizes where they change route, against the FP64 oracle or against
the same work done another way.  Tolerances are those of the operators' own parity tests: 1e-5
relative L2 for FP32 operators, bitwise where only the order of launches differs."""
import math

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2603_28756_gb300 as tm  # noqa: E402

PRIOR = dict(p=1.2, q=2.0, c=0.01, sigma=0.1, lam=1.0)


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32).ravel()).cuda()


def host(t, shape):
    torch.cuda.synchronize()
    return t.double().cpu().numpy().reshape(shape)


# odd sides (scalar accesses), sides that end a thread's column pair, a block's 256 columns and a walk
# of 8 or 32 rows, and enough slices for the long walks
@pytest.mark.parametrize("S,Nc", [(1, 1), (2, 5), (1, 33), (1, 257), (2, 258), (305, 64), (330, 63)])
def test_upsample_routes(orc, S, Nc):
    c = np.random.default_rng(S + Nc).standard_normal((S, Nc, Nc)).astype(np.float32)
    ctx = tm.Context([tm.Group(N=64, angles=[0.0], n_slices=1)])
    f = host(ctx.upsample_lanczos3(dev(c), S, Nc), (S, 2 * Nc, 2 * Nc))
    ref = orc.lanczos_up(c.astype(np.float64))
    assert np.array_equal(f[:, ::2, ::2], c.astype(np.float64))
    assert np.max(np.abs(f - ref)) < 1e-5 * np.max(np.abs(ref))


# rows of the spreading matrix at the grid's centre: about 5 (FP32 paths) and 11 (R*g) entries per
# angle, so 40 angles end in the rows a warp ranks, 200 in those a block sorts in shared memory and
# 1000 in those it sorts in place
@pytest.mark.parametrize("na", [1, 40, 200, 1000])
def test_spreading_matrix_rows(orc, na):
    N = 64
    p = synth.volume(S=1, N=N, n_angles=na, n_ellipsoids=4, seed=na)
    outs = []
    for _ in range(2):  # the fill order differs from run to run, the sorted rows must not
        ctx = tm.Context([tm.Group(N=N, angles=list(p.theta), n_slices=1)])
        outs.append((ctx.adjoint(dev(p.sino)), ctx.build_operator(dev(p.sino))))
    ref = orc.adjoint(p.sino.astype(np.float64), N, p.theta)
    assert rel(host(outs[0][0], ref.shape), ref) < 1e-5
    assert rel(host(outs[0][1], ref.shape), ref) < 1e-6
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def test_many_groups_reduce_like_one(orc):
    # more groups than the finalize kernel reduces between two barriers
    specs = [(64, 1 + k % 3, 9 + k) for k in range(18)]
    groups, sinos = [], []
    for k, (N, S, na) in enumerate(specs):
        p = synth.volume(S=S, N=N, n_angles=na, n_ellipsoids=3, seed=70 + k)
        groups.append(tm.Group(N=N, angles=list(p.theta), n_slices=S))
        sinos.append(p.sino.ravel())
    big = tm.Context(groups)
    atg = big.build_operator(dev(np.concatenate(sinos)))
    x = torch.zeros_like(atg)
    big.reconstruct(x, atg, tm.Params(**PRIOR, max_iter=6))
    off = 0
    for k, (N, S, na) in enumerate(specs):
        n = S * N * N
        ctx = tm.Context([groups[k]])
        x1 = torch.zeros(n, dtype=torch.float32, device="cuda")
        ctx.reconstruct(x1, ctx.build_operator(dev(sinos[k])), tm.Params(**PRIOR, max_iter=6))
        torch.cuda.synchronize()
        assert torch.equal(x[off:off + n], x1), k
        off += n


# pass 3b: bands of four and of eight rows, one and several column blocks, one slice and several,
# small and very large differences (the shared reciprocal), p = q (no threshold term)
@pytest.mark.parametrize("N,S,p,scale", [(64, 3, 1.2, 1.0), (256, 2, 1.0, 1e6), (512, 3, 1.2, 1.0), (512, 1, 2.0, 1.0),
                                         (1024, 2, 1.0, 1e-3)])
def test_prior_bands(orc, N, S, p, scale):
    th = synth.angles(4)
    ctx = tm.Context([tm.Group(N=N, angles=list(th), n_slices=S)])
    ctx.build_operator(torch.zeros(S * 4 * N, device="cuda"))
    x = synth.random_image(np.random.default_rng(N + S), (S, N, N), scale)
    zero = torch.zeros(S * N * N, device="cuda")
    prm = dict(p=p, q=2.0, c=0.01, sigma=0.1)
    # the prior alone: the gradient with it minus the gradient without, lambda so large that the
    # data term's rounding does not count
    lam = 1e12
    G = host(ctx.gradient(dev(x), zero, tm.Params(**prm, lam=lam)), x.shape)
    G0 = host(ctx.gradient(dev(x), zero, tm.Params(**prm, lam=0.0)), x.shape)
    ref = orc.prior(x.astype(np.float64), orc.Prior(**prm, lam=lam))[0]
    assert rel(G - G0, ref) < 1e-5


def _prior_gradient(x, prm, lam):
    S, N = x.shape[0], x.shape[1]
    ctx = tm.Context([tm.Group(N=N, angles=list(synth.angles(4)), n_slices=S)])
    ctx.build_operator(torch.zeros(S * 4 * N, device="cuda"))
    zero = torch.zeros(S * N * N, device="cuda")
    G = host(ctx.gradient(dev(x), zero, tm.Params(**prm, lam=lam, L=1.0)), x.shape)
    return G - host(ctx.gradient(dev(x), zero, tm.Params(**prm, lam=0.0, L=1.0)), x.shape)


# pass 3b: differences of up to 2^66 times c sigma, and around 2^62 times (where the two halves of a pair
# stop sharing a reciprocal), everywhere and in every second band only.  The exponent of
# r = 1 / (1 + 2^s) has an error of about 2^-24 s, s <= 66: 4e-6 of the pair's value
@pytest.mark.parametrize("N,p,sigma,scale", [(64, 1.0, 1e-18, 1.0), (512, 1.0, 1e-18, 1.0), (512, 1.0, 2.2e-17, 1.0),
                                             (512, 1.2, 1e-18, 1e4), (128, 1.2, 1e-18, 1e4)])
@pytest.mark.parametrize("mixed", [False, True])
def test_prior_at_huge_differences(orc, N, p, sigma, scale, mixed):
    S, R = 2, 8 if N >= 512 else 4
    x = synth.random_image(np.random.default_rng(N), (S, N, N), scale).astype(np.float32)
    r = np.arange(N)
    small = (r // R) % 2 == 1 if mixed else np.zeros(N, bool)
    x[:, small] *= np.float32(1e-12)
    prm = dict(p=p, q=2.0, c=0.01, sigma=sigma)
    lam = 1e12 * sigma  # the data term's rounding does not count
    G = _prior_gradient(x, prm, lam)
    ref = orc.prior(x.astype(np.float64), orc.Prior(**prm, lam=lam))[0]
    assert rel(G[:, ~small], ref[:, ~small]) < 1e-5
    if mixed:  # the rows whose neighbours are all small
        inner = small & (r % R > 0) & (r % R < R - 1)
        assert rel(G[:, inner], ref[:, inner]) < 1e-5


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_prior_keeps_a_bad_voxel_to_its_neighbours(bad):
    # the data term spreads it over its slice; in the slices before and after only the prior reads it
    S, N, r, c = 3, 512, 37, 131
    x = synth.random_image(np.random.default_rng(3), (S, N, N)).astype(np.float32)
    x[1, r, c] = bad
    G = _prior_gradient(x, dict(p=1.2, q=2.0, c=0.01, sigma=0.1), 1.0)
    want = np.zeros((N, N), bool)
    want[r - 1:r + 2, c - 1:c + 2] = True
    for z in (0, 2):
        assert np.array_equal(~np.isfinite(G[z]), want)


def test_operator_error_at_1536():
    # the transforms of this side came with 2.58e-7 from their first form (four radix stages) on these
    # inputs, its error against 64 bits; any other form has to stay there
    N, S, na = 1536, 4, 64
    ctx = tm.Context([tm.Group(N=N, angles=[math.pi * a / na for a in range(na)], n_slices=S)])
    ctx.build_operator(torch.zeros(S * na * N, device="cuda"))
    K = ctx.kernel(0).reshape(2 * N - 1, 2 * N - 1)
    torch.cuda.synchronize()
    C = torch.zeros(2 * N, 2 * N, device="cuda", dtype=torch.float64)
    i = torch.arange(-(N - 1), N, device="cuda") % (2 * N)
    C[i[:, None], i[None, :]] = K
    spec = torch.fft.rfft2(C).real
    errs = []
    for seed in (0, 1):
        x = torch.randn(S, N, N, device="cuda", generator=torch.Generator(device="cuda").manual_seed(seed))
        z = ctx.normal_apply(x.reshape(-1)).reshape(S, N, N).double()
        ref = torch.fft.irfft2(torch.fft.rfft2(x.double(), s=(2 * N, 2 * N)) * spec, s=(2 * N, 2 * N))[:, :N, :N]
        errs.append(float((z - ref).norm() / ref.norm()))
    assert np.mean(errs) < 2.58e-7, errs


# the general exponent in the bands of four and of eight rows, with several column blocks (pairs across a
# block's outer columns) and chunks of slices
@pytest.mark.parametrize("N,S,p,q", [(256, 2, 1.1, 1.8), (512, 3, 1.1, 1.8), (512, 2, 1.5, 3.0), (1024, 5, 1.2, 1.8)])
def test_prior_bands_general_q(orc, N, S, p, q):
    x = synth.random_image(np.random.default_rng(N + S), (S, N, N))
    prm = dict(p=p, q=q, c=0.01, sigma=0.1)
    G = _prior_gradient(x, prm, 1e12)
    ref = orc.prior(x.astype(np.float64), orc.Prior(**prm, lam=1e12))[0]
    assert rel(G, ref) < 1e-5


# R*g beside the bound that its FP32 storage sets (2.5e-8 of the norm): several hundred angles, whose rows at
# the grid's centre are shared by a warp, and the corner pixels, whose deconvolution factors are the largest
# and where the spreading kernel's own error, about 1e-7, is too
def test_atg_error_and_corners(orc):
    na = 400
    for N in (128, 1024):
        p = synth.volume(S=1, N=N, n_angles=na, n_ellipsoids=4, seed=N)
        g = p.sino.astype(np.float64)
        ctx = tm.Context([tm.Group(N=N, angles=list(p.theta), n_slices=1)])
        atg = host(ctx.build_operator(dev(p.sino)), (N, N))
        rms = np.sqrt(np.mean(atg ** 2))
        if N == 128:
            assert rel(atg, orc.adjoint(g, N, p.theta)[0]) < 5e-8
        at = [0, 1, 2, 3, N - 4, N - 3, N - 2, N - 1]
        err = max(abs(atg[r, c] - orc.adjoint_point(g[0], N, p.theta, r, c)) for r in at for c in at)
        assert err < 2.5e-7 * rms, (N, err / rms)
