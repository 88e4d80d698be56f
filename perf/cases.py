"""Performance cases: what users of this library have it do, through its public entry points.

A case is a dict of plain values; `prepare` makes what a user's program holds before the call (the
handle, its buffers, masks and uploaded arrays), `run` is one pass, `work` its unavoidable bytes and
operations, and `exact` the same outputs in 64 bits from plain torch.

Units are those of the library's workloads: 20 um sampling and 633 nm unless a case varies them.
The sources have a coherence width near one sample, so that the propagated light fills the grid and
mu is defined everywhere."""
import math
import random

import torch

import paper_2203_02734_gb300 as pw
from paper_2203_02734_gb300.autograd import CSDPropagation, GSMPropagation

D, LAM = 20e-6, 633e-9
FFT_N = (12, 16, 24, 32, 48, 64, 96, 128)  # grid sizes with an FFT plan


def listed():
    return [
        # the allocation-free call on the smallest grid of a latency-critical loop
        dict(name="noalloc_n16", kind="noalloc", N=16, z=0.5, aperture=True, lens=False, mask="none"),
        # one small interactive propagation: GSM source, W, S and mu
        dict(name="gsm_n32", kind="gsm", N=32, Nz=0, z=0.5, far=False, aperture=False, lens=False, mask="none"),
        # a multi-plane system: source, lens and finite pupil in an intermediate plane, image plane
        dict(name="chain_n64", kind="chain", N=64, z=0.3, z2=0.5, pupil=0.35),
        # a CSD exported by an earlier run, through a pupil mask, to the far field
        dict(name="uploaded_n96", kind="array", N=96, Nz=0, z=0.5, far=True, hermitian=True, mask="amp"),
        # an incoherent annulus in the far field (van Cittert-Zernike)
        dict(name="annulus_n128", kind="diagonal", N=128, z=2.0, far=True),
        # one step of the amplitude-mask inverse problem: forward and backward of a loss on S and mu
        dict(name="inverse_gsm_n96", kind="grad_gsm", N=96, z=1.0, far=False, loss="smu"),
        # forward and backward with the gradient of a whole uploaded CSD
        dict(name="inverse_csd_n48", kind="grad_csd", N=48, z=0.5, far=False, hermitian=True),
        # the focused beam through an aperture
        dict(name="aperture_lens_n128", kind="gsm", N=128, Nz=0, z=0.3, far=False, aperture=True, lens=True, mask="none"),
        # the largest grid: GSM light through a random phase screen
        dict(name="phase_screen_n256", kind="gsm", N=256, Nz=0, z=0.5, far=False, aperture=False, lens=False, mask="phase"),
        # the paper's zero-padded size, with the phase screen
        dict(name="padded_n200", kind="gsm", N=200, Nz=512, z=0.5, far=False, aperture=False, lens=False, mask="phase"),
        # a ragged grid without an FFT plan: an uploaded, general (non-Hermitian) array
        dict(name="ragged_n90", kind="array", N=90, Nz=0, z=0.4, far=False, hermitian=False, mask="phase"),
        # the polychromatic batch: 16 frequencies x 4 distances x 3 grid sizes, S and mu of each
        dict(name="polychromatic_batch", kind="batch", Ns="64,96,128", zs="0.1,0.5,1.0,5.0", freqs=16, aperture=False, keep=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["noalloc", "gsm", "gsm", "chain", "array", "diagonal", "grad_gsm", "grad_csd", "padded", "ragged", "batch"])
    z = round(_log(rng, 0.15, 2.0), 4)
    far, flag = rng.random() < 0.3, lambda: rng.random() < 0.5
    mask = rng.choice(["none", "phase", "amp"])
    if kind == "noalloc":
        return dict(kind=kind, N=rng.choice([8, 12, 16, 24, 32]), z=z, aperture=flag(), lens=flag(), mask=mask)
    if kind == "gsm":
        return dict(kind=kind, N=rng.choice(FFT_N + (128, 256)), Nz=0, z=z, far=far, aperture=flag(), lens=flag(), mask=mask)
    if kind == "chain":
        return dict(kind=kind, N=rng.choice(FFT_N), z=z, z2=round(_log(rng, 0.15, 2.0), 4), pupil=round(rng.uniform(0.25, 0.5), 3))
    if kind == "array":
        return dict(kind=kind, N=rng.choice(FFT_N), Nz=0, z=z, far=far, hermitian=flag(), mask=mask)
    if kind == "diagonal":
        return dict(kind=kind, N=rng.choice(FFT_N), z=z, far=far)
    if kind == "grad_gsm":
        return dict(kind=kind, N=rng.choice(FFT_N[2:]), z=z, far=far, loss=rng.choice(["s", "smu"]))
    if kind == "grad_csd":
        return dict(kind=kind, N=rng.choice(FFT_N[:7]), z=z, far=far, hermitian=flag())
    if kind == "padded":
        n = 2 * int(_log(rng, 8, 80))
        return dict(kind="gsm", N=n, Nz=n + 2 * int(n * rng.uniform(0.2, 0.9)), z=z, far=far, aperture=flag(), lens=flag(), mask=mask)
    if kind == "ragged":
        n = 2 * int(_log(rng, 9, 60))
        if n in FFT_N:
            n += 2
        return dict(kind="array", N=n, Nz=rng.choice([0, n + 2 * int(n * 0.3)]), z=z, far=far, hermitian=flag(), mask=mask)
    ns = sorted(rng.sample([16, 32, 64, 96, 128], rng.choice([1, 2])))
    return dict(kind="batch", Ns=",".join(map(str, ns)), zs=",".join(str(round(_log(rng, 0.15, 3.0), 3)) for _ in range(rng.choice([1, 2, 3]))),
                freqs=rng.choice([3, 8, 16]), aperture=flag(), keep=flag() and max(ns) <= 64)


# ---- inputs --------------------------------------------------------------------------------------

def _gsm(seed):
    r = random.Random(seed)
    return r.uniform(0.08e-3, 0.12e-3), r.uniform(14e-6, 20e-6), r.uniform(0.5, 1.5)


def _rand(seed, *shape):
    return torch.rand(*shape, generator=torch.Generator().manual_seed(seed), dtype=torch.float64).cuda()


def _blur(t, px):
    """Periodic Gaussian blur of the last two axes (std px samples)."""
    f = torch.fft.fftfreq(t.shape[-1], dtype=torch.float64, device=t.device)
    h = torch.exp(-2 * (math.pi * px * f) ** 2)
    return torch.fft.ifft2(torch.fft.fft2(t) * h[:, None] * h[None, :])


def _mask(kind, N, seed):
    """A phase screen correlated over three samples, or an amplitude mask in [0.5, 1] (complex64)."""
    if kind == "none":
        return None
    if kind == "amp":
        return (0.5 + 0.5 * _rand(seed, N, N)).to(torch.complex64)
    t = _blur(torch.exp(2j * math.pi * _rand(seed, N, N)), 3.0)
    return (t / t.abs()).to(torch.complex64)


def _array(N, seed, hermitian):
    """A CSD of eight random modes; without `hermitian`, a general array of the same kind."""
    g = _rand(seed, 4, 8, N, N) - 0.5
    u = _blur(torch.complex(g[0], g[1]), 0.6).reshape(8, N * N)
    v = u if hermitian else _blur(torch.complex(g[2], g[3]), 0.6).reshape(8, N * N)
    w = (0.5 + torch.arange(8, device="cuda", dtype=torch.float64) / 8)[:, None]
    return (torch.conj(u * w).T.to(torch.complex64) @ v.to(torch.complex64)).reshape(N, N, N, N).contiguous()


def _annulus(N, seed):
    n = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    r2 = n[:, None] ** 2 + n[None, :] ** 2
    r = random.Random(seed)
    ro = r.uniform(0.15, 0.3) * N
    ring = ((r2 <= ro * ro) & (r2 >= (0.4 * ro) ** 2)).to(torch.float64)
    return (ring * (0.5 + 0.5 * _rand(seed, N, N))).to(torch.float32)


def _places(case):
    """(aperture radius, focal length) in metres, 0 for none."""
    return 0.4 * case["N"] * D if case.get("aperture") else 0.0, case["z"] if case.get("lens") else 0.0


def _p1(N):
    return N // 2 - N // 8, N // 2 + 1


def _frequencies(n):
    """Wavelengths and Gaussian weights of a spectrum around 600 nm, 100 nm wide."""
    w0 = 2 * math.pi * 299792458.0 / 600e-9
    sw = w0 * (100e-9 / 600e-9) / 2.3548200450309493
    om = [w0 + sw * (-2 + 4 * k / max(n - 1, 1)) for k in range(n)]
    return [2 * math.pi * 299792458.0 / o for o in om], [math.exp(-((o - w0) / sw) ** 2 / 2) for o in om]


def _instances(case, seed):
    lams, wts = _frequencies(case["freqs"])
    sS, sM, A = _gsm(seed)
    for N in (int(x) for x in case["Ns"].split(",")):
        for z in (float(x) for x in case["zs"].split(",")):
            for lam, wt in zip(lams, wts):
                yield N, lam, z, sS, sM, A * wt, 0.4 * N * D if case["aperture"] else 0.0


class _Batch:
    """A batch with its workspace and outputs, destroyed with the object."""

    def __init__(self, case, seed):
        todo = list(_instances(case, seed))
        self.out = {}
        for N in sorted({t[0] for t in todo}):
            n = sum(t[0] == N for t in todo)
            self.out["S%d" % N] = torch.empty(n, N, N, dtype=torch.float32, device="cuda")
            self.out["mu%d" % N] = torch.empty(n, N, N, dtype=torch.complex64, device="cuda")
            if case["keep"]:
                self.out["W%d" % N] = torch.empty(n, N, N, N, N, dtype=torch.complex64, device="cuda")
        inst, at = [], {}
        for N, lam, z, sS, sM, A, radius in todo:
            k = at[N] = at.get(N, -1) + 1
            q = pw.pw_instance()
            q.N, q.dxi_m, q.lambda_m, q.z_m, q.farfield = N, D, lam, z, 0
            q.sigma_S_m, q.sigma_mu_m, q.amplitude, q.aperture_m, q.lens_f_m = sS, sM, A, radius, 0.0
            q.iP, q.jP = _p1(N)
            q.dev_S, q.dev_mu = self.out["S%d" % N][k].data_ptr(), self.out["mu%d" % N][k].data_ptr()
            if case["keep"]:
                q.dev_W = self.out["W%d" % N][k].data_ptr()
            inst.append(q)
        nb = pw.pw_batch_workspace_bytes(inst, 4)
        self.ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        self.b = pw.pw_batch_create(inst, 4, self.ws.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        if getattr(self, "b", None):
            pw.pw_batch_destroy(self.b)


def prepare(case, seed):
    N, kind = case.get("N"), case["kind"]
    s = dict(case=case, gsm=_gsm(seed))
    if kind == "batch":
        s["batch"] = _Batch(case, seed)
        return s
    if kind == "noalloc":
        s["W"] = torch.empty(N, N, N, N, dtype=torch.complex64, device="cuda")
        s["S"] = torch.empty(N, N, dtype=torch.float32, device="cuda")
        s["mask"] = _mask(case["mask"], N, seed)
        return s
    if kind == "grad_gsm":
        s["model"] = GSMPropagation(N, D, LAM, case["z"], P1=_p1(N), farfield=case["far"])
        s["p"] = [torch.tensor(v, dtype=torch.float32, requires_grad=True) for v in s["gsm"]]
        s["p"].append((0.5 + 0.5 * _rand(seed, N, N)).to(torch.float32).requires_grad_())
        s["target"] = _targets(case, seed)
        return s
    if kind == "grad_csd":
        s["model"] = CSDPropagation(N, D, LAM, case["z"], P1=_p1(N), farfield=case["far"], hermitian=case["hermitian"])
        s["W0"] = _array(N, seed, True).requires_grad_()
        s["target"] = _targets(case, seed)
        return s
    s["csd"] = pw.CSD(N, D, LAM)
    if case.get("Nz"):
        pw.pw_csd_set_padding(s["csd"].h, case["Nz"])
    s["mask"] = _mask(case.get("mask", "none"), N, seed)
    if kind == "array":
        s["W0"] = _array(N, seed, case["hermitian"])
    if kind == "diagonal":
        s["d"] = _annulus(N, seed)
    return s


def _targets(case, seed):
    """The measured S and mu of an inverse problem (those of a known source near the sought one)."""
    N = case["N"]
    S, mu = _gsm_s_mu(N, D, LAM, case["z"], case["far"], *_gsm(seed + 1), None, N)
    if case["kind"] == "grad_csd":  # a flat S of the power that the uploaded CSD carries
        power = torch.diagonal(_array(N, seed, True).reshape(N * N, N * N)).real.double().sum()
        S = torch.ones_like(S) * power * (D * D / (LAM * case["z"])) ** 2
    return S.to(torch.float32), mu.to(torch.complex64), float((1.0 / S.max()).item())


def _loss(case, S, mu, target):
    St, mut, unit = target
    loss = (((S - St) * unit) ** 2).sum()
    if case.get("loss", "smu") == "smu":
        w = St * unit
        loss = loss + (w * ((mu - mut).real ** 2 + (mu - mut).imag ** 2)).sum()
    return loss


# ---- one pass ------------------------------------------------------------------------------------

def run(s):
    case, kind = s["case"], s["case"]["kind"]
    N = case.get("N")
    if kind == "batch":
        pw.pw_batch_run(s["batch"].b)
        return s["batch"].out
    if kind == "noalloc":
        radius, f = _places(case)
        m = s["mask"]
        pw.pw_propagate_gsm_fresnel_noalloc(N, D, LAM, case["z"], *s["gsm"], radius, f, 0 if m is None else m.data_ptr(),
                                            s["W"].data_ptr(), s["W"].numel() * 8, s["S"].data_ptr(),
                                            torch.cuda.current_stream().cuda_stream)
        return [s["W"], s["S"]]
    if kind == "grad_gsm":
        for p in s["p"]:
            p.grad = None
        S, mu = s["model"](*s["p"])
        _loss(case, S, mu, s["target"]).backward()
        return [S, mu] + [p.grad for p in s["p"]]
    if kind == "grad_csd":
        s["W0"].grad = None
        S, mu = s["model"](s["W0"])
        _loss(case, S, mu, s["target"]).backward()
        return [S, mu, s["W0"].grad]
    c = s["csd"]
    c.reset(D)
    if kind == "array":
        c.source_array(s["W0"], case["hermitian"])
    elif kind == "diagonal":
        pw.pw_source_diagonal(c.h, s["d"].data_ptr(), 1.0)
    else:
        c.source_gsm(*s["gsm"])
    radius, f = _places(case)
    if radius:
        c.source_aperture(radius)
    if f:
        c.source_lens(f)
    if s["mask"] is not None:
        c.source_mask(s["mask"])
    (c.propagate_farfield if case.get("far") else c.propagate_fresnel)(case["z"])
    if kind == "chain":
        c.source_lens(0.7 * case["z2"])
        c.source_aperture(case["pupil"] * N * c.sampling())
        c.propagate_fresnel(case["z2"])
        return [c.W, c.spectral_density()]
    if not case.get("hermitian", True):  # mu is defined for a CSD
        return [c.W, c.spectral_density()]
    return [c.W, c.spectral_density(), c.degree_of_coherence(*_p1(N))]


def work(case):
    """Every input read once and every output written once; operations of the FFTs over the four
    axes of the whole array (three for a GSM source, whose factors separate one axis; the outer
    product alone for a delta-correlated source, whose propagated CSD depends on x1 - x2)."""
    kind = case["kind"]
    if kind == "batch":
        nb = fl = 0
        for N, *_ in _instances(case, 0):
            L = 4 * N * N
            nb += N * N * 12 + (8 * N ** 4 if case["keep"] else 0)
            fl += 15 * L * math.log2(L) + 16 * N ** 3 + (15 * N ** 4 * math.log2(N) if case["keep"] else 0)
        return dict(bytes=nb, flops=fl)
    N = case["N"]
    P, L = N ** 4, math.log2(max(case.get("Nz") or 0, N)) * max(case.get("Nz") or 0, N) / N
    nb, fl = 12 * N * N + 8 * N * N * (case.get("mask", "none") != "none"), 0.0
    if kind == "noalloc" or kind == "gsm":
        nb, fl = nb + 8 * P, 15 * P * L
    elif kind == "chain":
        nb, fl = nb + 8 * P, 35 * P * L
    elif kind == "array":
        nb, fl = nb + 16 * P, 20 * P * L
    elif kind == "diagonal":
        nb, fl = nb + 8 * P + 4 * N * N, 6 * P
    elif kind == "grad_gsm":  # S and mu forward; the adjoint source has 2 N^2 non-zeros
        nb, fl = nb + 32 * N * N, 30 * 4 * N * N * math.log2(4 * N * N) + 32 * N ** 3 + 10 * P
    else:
        nb, fl = nb + 16 * P + 20 * N * N, 12 * P
    return dict(bytes=nb, flops=fl)


# ---- the same in 64 bits, from plain torch ---------------------------------------------------------

def _axis(N, d, lam, z, far, Nz):
    """Kernel of one axis, N outputs x N inputs: q(X_k) exp(-2 pi i k n / Nz) q(x_n), centred indices."""
    n = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    dx = lam * z / (Nz * d)
    q = lambda t: torch.exp(2j * math.pi * torch.remainder(t, 1.0))  # noqa: E731
    kn = torch.remainder(n[:, None] * n[None, :], Nz) / Nz
    E = q(n[:, None] ** 2 * (dx * dx / (2 * lam * z))) * q(-kn)
    return (E if far else E * q(n[None, :] ** 2 * (d * d / (2 * lam * z)))), dx


def _propagate(W, d, lam, z, far, Nz):
    E, dx = _axis(W.shape[0], d, lam, z, far, Nz)
    for axis in (3, 2, 1, 0):
        W = torch.tensordot(E if axis > 1 else torch.conj(E), W, dims=([1], [axis])).movedim(0, axis)
    return W * (d * d / (lam * z)) ** 2, dx


def _planes(N, d, lam, radius, f, mask):
    """Aperture, thin lens and mask of a plane, as one N x N factor."""
    n = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    r2 = n[:, None] ** 2 + n[None, :] ** 2
    m = torch.ones(N, N, dtype=torch.complex128, device="cuda") if mask is None else mask.to(torch.complex128)
    if radius:
        m = m * (r2 <= (radius / d) ** 2)
    if f:
        m = m * torch.exp(-2j * math.pi * torch.remainder(r2 * (d * d / (2 * lam * f)), 1.0))
    return m


def _gsm_w0(N, sS, sM, A):
    x = (torch.arange(N, device="cuda", dtype=torch.float64) - N // 2) * D
    G = torch.exp(-(x[:, None] ** 2 + x[None, :] ** 2) / (4 * sS ** 2) - (x[:, None] - x[None, :]) ** 2 / (2 * sM ** 2))
    return A * G[:, None, :, None] * G[None, :, None, :]


def _s_mu(W, P):
    N = W.shape[0]
    M = W.reshape(N * N, N * N)
    S = torch.diagonal(M).real
    den = S[P[0] * N + P[1]] * S
    mu = torch.where(den > 0, M[P[0] * N + P[1]] * torch.rsqrt(torch.where(den > 0, den, torch.ones_like(den))), torch.zeros_like(M[0]))
    return S.reshape(N, N), mu.reshape(N, N)


def _gsm_s_mu(N, d, lam, z, far, sS, sM, A, m, Nz):
    """S and mu(P1, .) of the propagated GSM source without its CSD: S is the transform of the
    correlation of the source field with itself times the coherence, mu's row two matrix products."""
    n = torch.arange(N, device="cuda", dtype=torch.float64) - N // 2
    E, dx = _axis(N, d, lam, z, far, Nz)
    F = torch.ones(N, N, dtype=torch.complex128, device="cuda") if m is None else m
    h = torch.exp(-(n * d) ** 2 / (4 * sS ** 2))
    k = lambda u: torch.exp(-(u * d) ** 2 / (2 * sM ** 2))  # noqa: E731
    q = torch.ones(N, dtype=torch.complex128, device="cuda") if far else E[N // 2]  # input propagator (k = 0)
    P = F * h[:, None] * h[None, :] * q[:, None] * q[None, :]
    f = torch.fft.fft2(P, s=(2 * N, 2 * N))
    C = torch.fft.ifft2(f * torch.conj(f))  # sum_x conj(P(x)) P(x + u)
    u = torch.fft.fftfreq(2 * N, 1.0 / (2 * N), dtype=torch.float64, device="cuda")
    C = C * k(u)[:, None] * k(u)[None, :]
    B = torch.exp(-2j * math.pi * torch.remainder(n[:, None] * u[None, :], Nz) / Nz)
    s = A * (d * d / (lam * z)) ** 2
    S = s * (B @ C @ B.T).real
    G = h[:, None] * h[None, :] * k(n[:, None] - n[None, :])
    ip, jp = _p1(N)
    Q = torch.conj(F) * torch.conj(E[ip])[:, None] * torch.conj(E[jp])[None, :]
    row = s * (E @ (F * (G.T.to(Q.dtype) @ Q @ G.to(Q.dtype))) @ E.T)
    den = S[ip, jp] * S
    return S, torch.where(den > 0, row * torch.rsqrt(torch.where(den > 0, den, torch.ones_like(den))), torch.zeros_like(row))


def exact(case, seed):
    N, kind = case.get("N"), case["kind"]
    if kind == "batch":
        out = {}
        for n, lam, z, sS, sM, A, radius in _instances(case, seed):
            m = _planes(n, D, lam, radius, 0.0, None)
            S, mu = _gsm_s_mu(n, D, lam, z, False, sS, sM, A, m, n)
            out.setdefault("S%d" % n, []).append(S)
            out.setdefault("mu%d" % n, []).append(mu)
            if case["keep"]:
                W0 = _gsm_w0(n, sS, sM, A) * torch.conj(m)[:, :, None, None] * m
                out.setdefault("W%d" % n, []).append(_propagate(W0, D, lam, z, False, n)[0])
        return {k: torch.stack(v) for k, v in out.items()}
    z, far, Nz = case["z"], case.get("far", False), case.get("Nz") or N
    sS, sM, A = _gsm(seed)
    if kind == "grad_gsm":
        p = [torch.tensor(v, dtype=torch.float32, device="cuda").double().requires_grad_() for v in (sS, sM, A)]
        p.append((0.5 + 0.5 * _rand(seed, N, N)).to(torch.float32).double().requires_grad_())
        S, mu = _gsm_s_mu(N, D, LAM, z, far, p[0], p[1], p[2], p[3].to(torch.complex128), N)
        return [S.detach(), mu.detach()] + list(torch.autograd.grad(_loss(case, S, mu, _targets(case, seed)), p))
    if kind == "grad_csd":
        W0 = _array(N, seed, True).to(torch.complex128).requires_grad_()
        S, mu = _s_mu(_propagate(W0, D, LAM, z, far, N)[0], _p1(N))
        return [S.detach(), mu.detach(), torch.autograd.grad(_loss(case, S, mu, _targets(case, seed)), W0)[0]]
    mask = _mask(case.get("mask", "none"), N, seed)
    m = _planes(N, D, LAM, *_places(case), mask)
    if kind == "gsm" and N > 200:  # the whole CSD in 64 bits does not fit
        return [None] + list(_gsm_s_mu(N, D, LAM, z, far, sS, sM, A, m, Nz))
    if kind == "array":
        W0 = _array(N, seed, case["hermitian"]).to(torch.complex128)
    elif kind == "diagonal":
        W0 = torch.diag(_annulus(N, seed).double().reshape(-1)).reshape(N, N, N, N).to(torch.complex128)
    else:
        W0 = _gsm_w0(N, sS, sM, A).to(torch.complex128)
    W0 = W0 * torch.conj(m)[:, :, None, None]
    W0 *= m
    W, dx = _propagate(W0, D, LAM, z, far, Nz)
    del W0
    if kind == "chain":
        m = _planes(N, dx, LAM, case["pupil"] * N * dx, 0.7 * case["z2"], None)
        W = W * torch.conj(m)[:, :, None, None] * m
        W, dx = _propagate(W, dx, LAM, case["z2"], False, N)
    S, mu = _s_mu(W, _p1(N))
    return [W, S] if kind in ("noalloc", "chain") or not case.get("hermitian", True) else [W, S, mu]
