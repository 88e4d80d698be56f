"""The closed forms and the plane kernels at the sizes where their launch shapes differ: parameter gradients
(csrc/delta.cuh) with two columns a block (N = 2, 6), idle threads (N = 12, 24, 48) and one row of threads (N = 128, 256),
with and without a mu term, against torch's autograd in FP64; GSM and delta-correlated sources at N = 128 against the
same source as an uploaded array.

Bounds: R takes the FP32 rounding of its tables and factors, some 20 roundings of 2^-24 a term, all positive upstream
gradients of S; the terms add up in pairs of floats.  1e-5 of the mask gradient in L2 and of each parameter's
gradient leaves a factor of eight.  Two FP32 propagations differ by at most 2e-6 (see test_planes.py)."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from gpu_cases import rel

D, LAM = 20e-6, 633e-9


def s_mu(torch, N, z, far, sS, sM, A, a, P1):
    """S and mu of the amplitude-masked GSM source in FP64, differentiable."""
    n = torch.arange(N, dtype=torch.float64) - N // 2
    turns = lambda t: torch.exp(2j * np.pi * torch.remainder(t, 1.0))  # noqa: E731
    dx = LAM * z / (N * D)
    E = turns(n[:, None] ** 2 * (dx * dx / (2 * LAM * z))) * turns(-torch.remainder(n[:, None] * n[None, :], N) / N)
    q = torch.ones(N, dtype=torch.complex128) if far else turns(n ** 2 * (D * D / (2 * LAM * z)))
    h = torch.exp(-(n * D) ** 2 / (4 * sS ** 2))
    k = lambda u: torch.exp(-(u * D) ** 2 / (2 * sM ** 2))  # noqa: E731
    F = a * q[:, None] * q[None, :]
    Ph = torch.fft.fft2(F * h[:, None] * h[None, :], s=(2 * N, 2 * N))
    u = torch.fft.fftfreq(2 * N, 1.0 / (2 * N), dtype=torch.float64)
    C = torch.fft.ifft2(Ph * Ph.conj()) * k(u)[:, None] * k(u)[None, :]
    B = turns(-torch.remainder(n[:, None] * u[None, :], N) / N)
    s = A * (D * D / (LAM * z)) ** 2
    S = s * (B @ C @ B.T).real
    G = (h[:, None] * h[None, :] * k(n[:, None] - n[None, :])).to(torch.complex128)
    c1 = E[P1[0]].conj()[:, None] * E[P1[1]].conj()[None, :]
    row = s * E @ (F * (G @ (F.conj() * c1) @ G)) @ E.T
    return S, row / torch.sqrt(S[P1] * S)


def _upstream(N, S):
    r = np.random.default_rng(N)
    return (0.5 + r.random((N, N))) / float(S.max()), (r.normal(size=(N, N)) + 1j * r.normal(size=(N, N))) * 0.1


def _reference(torch, N, z, far, gsm, a, P1, with_mu):
    p = [torch.tensor(float(np.float32(v)), dtype=torch.float64, requires_grad=True) for v in gsm]
    p.append(torch.from_numpy(a.astype(np.float64)).requires_grad_())
    S, mu = s_mu(torch, N, z, far, *p, P1)
    gS, gmu = _upstream(N, S.detach())
    loss = (torch.from_numpy(gS) * S).sum()
    if with_mu:
        loss = loss + (torch.from_numpy(gmu).conj() * mu).real.sum()
    return S.detach().numpy(), mu.detach().numpy(), [g.numpy() for g in torch.autograd.grad(loss, p)], (gS, gmu)


@pytest.mark.parametrize("N,far", [(6, False), (8, True)])
def test_reference_against_the_oracle(N, far):
    torch = pytest.importorskip("torch")
    a, P1, gsm = WL.amplitude_mask(N, seed=3).real, (N // 2 - 1, N - 1), (3 * D, 1.2 * D, 0.9)
    S, mu, _, _ = _reference(torch, N, 0.3, far, gsm, a, P1, True)
    W, _ = O.propagate_fft(O.apply_mask(O.gsm_source(N, D, *[float(np.float32(v)) for v in gsm]), a), D, LAM, 0.3, farfield=far)
    assert rel(S, O.spectral_density(W).real) < 1e-12
    assert rel(mu, O.degree_of_coherence(W, *P1)) < 1e-10


@pytest.mark.gpu
@pytest.mark.parametrize("N", [2, 4, 6, 12, 24, 48, 96, 128, 256])
@pytest.mark.parametrize("with_mu", [False, True])
@pytest.mark.parametrize("far", [False, True])
def test_parameter_gradients(N, with_mu, far):
    import torch
    from paper_2203_02734_gb300.autograd import GSMPropagation
    a, P1, gsm, z = WL.amplitude_mask(N, seed=3).real.astype(np.float32), (N // 2 - 1, N // 2), (max(N / 6, 0.8) * D, 1.1 * D, 0.9), 0.4
    _, _, ref, (gS, gmu) = _reference(torch, N, z, far, gsm, a, P1, with_mu)
    p = [torch.tensor(v, dtype=torch.float32, device="cuda").requires_grad_() for v in gsm]
    p.append(torch.from_numpy(a).cuda().requires_grad_())
    model = GSMPropagation(N, D, LAM, z, P1=P1, farfield=far)
    S, mu = model(*p)
    loss = (torch.from_numpy(gS).to(torch.float32).cuda() * S).sum()
    if with_mu:
        loss = loss + (torch.from_numpy(gmu).to(torch.complex64).cuda().conj() * mu).real.sum()
    loss.backward()
    model.close()
    for x, r, v in zip(p[:3], ref, gsm):  # in units of each parameter: sigma_mu's terms cancel, A's are positive
        assert abs(float(x.grad) - float(r)) * v < 1e-5 * abs(float(ref[2])) * gsm[2]
    assert rel(p[3].grad.cpu().numpy().astype(np.float64), ref[3]) < 1e-5


def _against_array(source, W0, N, far, setup):
    import paper_2203_02734_gb300 as pw
    out = []
    for array in (False, True):
        c = pw.CSD(N, D, LAM)
        c.source_array(W0) if array else source(c, pw)
        setup(c)
        (c.propagate_farfield if far else c.propagate_fresnel)(0.3)
        out.append((c.W, c.spectral_density()))
        pw.pw_csd_check(c.h)
        c.close()
    for x, y in zip(*out):
        num = sum(float((x[a] - y[a]).abs().double().square().sum()) for a in range(N))
        den = sum(float(y[a].abs().double().square().sum()) for a in range(N))
        assert (num / den) ** 0.5 < 2e-6


@pytest.mark.gpu
@pytest.mark.parametrize("far", [False, True])
def test_planes_n128_against_the_general_passes(far):
    import torch
    N = 128
    x = (torch.arange(N, device="cuda", dtype=torch.float64) - N // 2) * D
    G = torch.exp(-(x[:, None] ** 2 + x[None, :] ** 2) / (4 * (12 * D) ** 2) - (x[:, None] - x[None, :]) ** 2 / (2 * (1.5 * D) ** 2))
    W0 = torch.stack([(0.8 * G[a][None, :, None] * G[:, None, :]).to(torch.complex64) for a in range(N)])
    m = torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=3))).cuda()

    def setup(c):
        c.source_mask(m)
        c.source_aperture(0.4 * N * D)
        c.source_lens(0.5)
    _against_array(lambda c, pw: c.source_gsm(12 * D, 1.5 * D, 0.8), W0, N, far, setup)


@pytest.mark.gpu
@pytest.mark.parametrize("far", [False, True])
def test_diagonal_n128_against_the_general_passes(far):
    import torch
    N = 128
    d = torch.rand(N, N, device="cuda", generator=torch.Generator(device="cuda").manual_seed(N)) - 0.2
    W0 = torch.zeros(N * N, N * N, dtype=torch.complex64, device="cuda")
    W0.diagonal().copy_(0.7 * d.reshape(-1))
    _against_array(lambda c, pw: pw.pw_source_diagonal(c.h, d.data_ptr(), 0.7), W0.reshape(N, N, N, N), N, far,
                   lambda c: c.source_aperture(0.45 * N * D))


@pytest.mark.gpu
@pytest.mark.parametrize("N", [48, 64, 96, 128])
def test_general_store_against_the_hermitian_one(N):
    import torch
    import paper_2203_02734_gb300 as pw
    g = torch.Generator(device="cuda").manual_seed(N)
    u = torch.randn(N * N, 4, dtype=torch.complex64, device="cuda", generator=g)
    W0 = (u.conj() @ u.T).reshape(N, N, N, N)
    out = []
    for hermitian in (False, True):
        c = pw.CSD(N, D, LAM)
        c.source_array(W0, hermitian)
        c.source_aperture(0.45 * N * D)
        c.propagate_fresnel(0.3)
        out.append((c.W, c.spectral_density()))
        c.close()
    for x, y in zip(*out):
        assert float(torch.linalg.vector_norm(x - y)) < 2e-6 * float(torch.linalg.vector_norm(y))
