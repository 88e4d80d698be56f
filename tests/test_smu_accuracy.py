"""Point by point accuracy of S and mu of a GSM source without its CSDA (csrc/smu.cuh), dim regions and corner P1
included, against FP64.

Both arithmetics (FP64, float pairs of 48 bits) leave the rounding of the FP32 outputs and an error of the
transforms relative to the brightest point: with L = 512 the sums over (2N)^2 points of values good to 2^-44
err by at most some 2^-44 x 16 = 2^-40 of max S.  mu = row / sqrt(S(P1) S(x)) takes half the error of each rounded S
(2^-24 in all), 2^-22 of the reciprocal root (2 ulp), 2^-23 of products and conversions, and the transforms'
error, 2^-40 max S / sqrt(S(P1) S(x)) in units of mu; the errors of S there count likewise."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from gpu_cases import rel

D, LAM = 20e-6, 633e-9


def exact(N, lam, z, far, sS, sM, A, ap, f, m, P1):
    """S and mu in FP64: the transform of the field's correlation times its coherence, and the row of P1."""
    n = np.arange(N) - N // 2
    turns = lambda t: np.exp(2j * np.pi * np.remainder(t, 1.0))  # noqa: E731
    dx = lam * z / (N * D)
    E = turns(n[:, None] ** 2 * (dx * dx / (2 * lam * z))) * turns(-np.remainder(n[:, None] * n[None, :], N) / N)
    q = turns(n ** 2 * (D * D / (2 * lam * z))) if not far else np.ones(N)
    lens = turns(-n ** 2 * (D * D / (2 * lam * f))) if f else np.ones(N)
    F = np.ones((N, N)) if m is None else m.astype(complex)
    if ap:
        F = F * ((n[:, None] ** 2 + n[None, :] ** 2) <= (ap / D) ** 2)
    F = F * (q * lens)[:, None] * (q * lens)[None, :]
    h = np.exp(-(n * D) ** 2 / (4 * sS ** 2))
    k = lambda u: np.exp(-(u * D) ** 2 / (2 * sM ** 2))  # noqa: E731
    P = F * h[:, None] * h[None, :]
    u = np.fft.fftfreq(2 * N, 1.0 / (2 * N))
    C = np.fft.ifft2(np.abs(np.fft.fft2(P, s=(2 * N, 2 * N))) ** 2) * k(u)[:, None] * k(u)[None, :]
    B = turns(-np.remainder(n[:, None] * u[None, :], N) / N)
    s = A * (D * D / (lam * z)) ** 2
    S = s * (B @ C @ B.T).real
    G = h[:, None] * h[None, :] * k(n[:, None] - n[None, :])
    c1 = np.conj(E[P1[0]])[:, None] * np.conj(E[P1[1]])[None, :]  # the output kernel of P1
    row = s * E @ (F * (G @ (np.conj(F) * c1) @ G)) @ E.T
    den = S[P1] * S
    return S, np.where(den > 0, row / np.sqrt(np.where(den > 0, den, 1.0)), 0)


@pytest.mark.parametrize("N,far,P1", [(6, False, (0, 5)), (8, True, (7, 2)), (12, False, (6, 4))])
def test_reference_against_the_oracle(N, far, P1):
    m = WL.to_c64(WL.phase_screen(N, seed=5, corr_px=1.0))
    ap, f = 0.45 * N * D, 0.4
    m1 = m.astype(complex) * O.circle_aperture(N, D, ap) * O.thin_lens(N, D, LAM, f)
    W, _ = O.propagate_fft(O.apply_mask(O.gsm_source(N, D, 3 * D, 1.5 * D, 0.7), m1), D, LAM, 0.3, farfield=far)
    S, mu = exact(N, LAM, 0.3, far, 3 * D, 1.5 * D, 0.7, ap, f, m, P1)
    assert rel(S, O.spectral_density(W).real) < 1e-12
    assert rel(mu, O.degree_of_coherence(W, *P1)) < 1e-11


def _check(S, mu, ref):
    Sr, mr, P1 = ref
    S, mu = S.cpu().numpy().astype(np.float64), mu.cpu().numpy().astype(np.complex128)
    top = Sr.max()
    assert (np.abs(S - Sr) <= 2.0 ** -24 * 1.01 * Sr + 2.0 ** -40 * top).all()
    assert Sr[P1] >= 1e-6 * top  # mu is compared for this P1
    lit = Sr >= 1e-6 * top
    bound = 2.0 ** -24 + 2.0 ** -22 + 2.0 ** -23 + 2.0 ** -39 * top / np.sqrt(Sr[P1] * np.where(lit, Sr, top))
    assert (np.abs(mu - mr) <= bound)[lit].all()


# (sigma_S, sigma_mu in pixels, aperture, lens, mask): light that fills the output grid, coherence over several pixels
# with and without a hard edge (S falls to 1e-6 of its maximum and below), nearly coherent light
SOURCES = [(5, 0.6, False, False, True), (5, 2, False, False, False), (15, 5, False, True, False), (5, 5, True, True, False),
           (15, 60, True, False, True), (8, 0.6, True, False, False)]


def _places(N):
    return [(0, N - 1), (N // 2, N // 3), (N - 1, 2)]


def _reference(N, i, lam, z, far):
    """Reference of source i with the first P1 that is lit at all."""
    sS, sM, ap, lens, mask = SOURCES[i]
    m = WL.to_c64(WL.phase_screen(N, seed=7)) if mask else None
    args = (sS * D, sM * D, 0.8 + 0.1 * i, 0.4 * N * D if ap else 0.0, 0.4 if lens else 0.0)
    for P1 in _places(N)[i % 3:] + [(N // 2, N // 2 - 1)]:
        S, mu = exact(N, lam, z, far, *args, m, P1)
        if S[P1] >= 1e-6 * S.max():
            return args, m, (S, mu, P1)


def test_corners_are_compared():
    for N in (16, 32, 64, 96, 128):
        assert [_reference(N, i, LAM, 0.3, False)[2][2] for i in (0, 5)] == [(0, N - 1), (N - 1, 2)]


@pytest.mark.gpu
@pytest.mark.parametrize("N,pool", [(16, 1), (32, 2), (64, 1), (96, 2), (128, 1)])
@pytest.mark.parametrize("far", [False, True])
def test_batch_point_by_point(N, pool, far):
    import torch
    import paper_2203_02734_gb300 as pw
    n = len(SOURCES)
    S = torch.full((n, N, N), float("nan"), device="cuda")
    mu = torch.full((n, N, N), float("nan"), dtype=torch.complex64, device="cuda")
    insts, refs, keep = [], [], []
    for i in range(n):
        lam, z = LAM * (1 + 0.02 * i), 0.3 + 0.05 * i
        (sS, sM, A, ap, f), m, ref = _reference(N, i, lam, z, far)
        refs.append(ref)
        q = pw.pw_instance()
        q.N, q.dxi_m, q.lambda_m, q.z_m, q.farfield = N, D, lam, z, int(far)
        q.sigma_S_m, q.sigma_mu_m, q.amplitude, q.aperture_m, q.lens_f_m = sS, sM, A, ap, f
        if m is not None:
            keep.append(torch.from_numpy(m).cuda())
            q.dev_mask = keep[-1].data_ptr()
        (q.iP, q.jP), q.dev_S, q.dev_mu = ref[2], S[i].data_ptr(), mu[i].data_ptr()
        insts.append(q)
    nb = pw.pw_batch_workspace_bytes(insts, pool)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    b = pw.pw_batch_create(insts, pool, ws.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)
    pw.pw_batch_run(b)
    pw.pw_batch_check(b)
    pw.pw_batch_destroy(b)
    for i in range(n):
        _check(S[i], mu[i], refs[i])


@pytest.mark.gpu
@pytest.mark.parametrize("N", [4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256])
@pytest.mark.parametrize("far", [False, True])
def test_handle_point_by_point(N, far):
    import torch
    import paper_2203_02734_gb300 as pw
    S = torch.empty(N, N, device="cuda")
    mu = torch.empty(N, N, dtype=torch.complex64, device="cuda")
    c = pw.CSD(N, D, LAM)
    for i in range(len(SOURCES)):
        (sS, sM, A, ap, f), m, ref = _reference(N, i, LAM, 0.3, far)
        c.reset(D)
        c.source_gsm(sS, sM, A)
        c.source_aperture(ap)
        c.source_lens(f)
        if m is not None:
            c.source_mask(torch.from_numpy(m).cuda())
        pw.pw_gsm_s_mu(c.h, 0.3, far, *ref[2], S.data_ptr(), mu.data_ptr())
        _check(S, mu, ref)
    c.close()


# N = 256: the planes' S and mu after the propagation are as accurate as the three passes that they replaced, whose
# relative L2 errors over these sources were 1.2e-7 and 1.9e-7 in the mean; 1.3e-7 and 2.2e-7 allow for the library's
# rounding elsewhere.
@pytest.mark.gpu
def test_planes_n256_are_as_accurate_as_the_passes():
    import torch
    import paper_2203_02734_gb300 as pw
    N, P1, eS, emu = 256, (256 // 2 - 256 // 8, 256 // 2 + 1), [], []
    c = pw.CSD(N, D, LAM)
    for i, (z, ap, m) in enumerate([(0.5, 0.0, WL.phase_screen(N, seed=1)), (0.3, 0.4 * N * D, None), (1.1, 0.0, WL.amplitude_mask(N, seed=3))]):
        args = (5 * D, (0.7 + 0.1 * i) * D, 0.6 + 0.3 * i)
        m = None if m is None else WL.to_c64(m)
        c.reset(D)
        c.source_gsm(*args)
        c.source_aperture(ap)
        if m is not None:
            c.source_mask(torch.from_numpy(m).cuda())
        c.propagate_fresnel(z)
        S, mu = exact(N, LAM, z, False, *args, ap, 0.0, m, P1)
        eS.append(rel(c.spectral_density().cpu().numpy().astype(np.float64), S))
        emu.append(rel(c.degree_of_coherence(*P1).cpu().numpy().astype(complex), mu))
    c.close()
    assert np.mean(eS) < 1.3e-7 and np.mean(emu) < 2.2e-7, (eS, emu)


# The range of FP32 has to hold S and W, not the amplitude or the masks by themselves: a strong source behind weak masks,
# and a strong one without, give the scaled result of an ordinary one (powers of two round nothing).
@pytest.mark.gpu
@pytest.mark.parametrize("N", [16, 32, 64, 96, 128])
@pytest.mark.parametrize("keep", [False, True])
def test_range_of_amplitude_and_mask(N, keep):
    import torch
    import paper_2203_02734_gb300 as pw
    m = torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=7))).cuda()
    P1, out = (N // 2, N // 2 - 1), []
    for A, w in [(1.0, 1.0), (2.0 ** 126, 2.0 ** -63), (-2.0 ** 110, 1.0)]:
        S = torch.empty(N, N, device="cuda")
        mu = torch.empty(N, N, dtype=torch.complex64, device="cuda")
        W = torch.empty((N,) * 4 if keep else (1,), dtype=torch.complex64, device="cuda")
        mask = m * w
        q = pw.pw_instance()
        q.N, q.dxi_m, q.lambda_m, q.z_m, q.sigma_S_m, q.sigma_mu_m, q.amplitude = N, D, LAM, 0.3, 5 * D, 1.5 * D, A
        (q.iP, q.jP), q.dev_S, q.dev_mu, q.dev_mask = P1, S.data_ptr(), mu.data_ptr(), mask.data_ptr()
        if keep:
            q.dev_W = W.data_ptr()
        nb = pw.pw_batch_workspace_bytes([q], 1)
        ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
        b = pw.pw_batch_create([q], 1, ws.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)
        pw.pw_batch_set_mode(b, pw.PW_BATCH_SEQUENCED)
        pw.pw_batch_run(b)
        pw.pw_batch_check(b)
        pw.pw_batch_destroy(b)
        c = pw.CSD(N, D, LAM)
        c.source_gsm(5 * D, 1.5 * D, A)
        c.source_mask(mask)
        Sh, muh = torch.empty_like(S), torch.empty_like(mu)
        pw.pw_gsm_s_mu(c.h, 0.3, False, *P1, Sh.data_ptr(), muh.data_ptr())
        c.propagate_fresnel(0.3)
        out.append((S, mu, W, Sh, muh, c.W, c.spectral_density()))
        c.close()
    for x, y, v in zip(*out):
        if x.numel() > 1:
            norm = float(torch.linalg.vector_norm(x))
            assert float(torch.linalg.vector_norm(x - y)) <= 3e-7 * norm
            if x.shape != mu.shape or not x.is_complex():  # not mu: S(P1) S(x) leaves the range
                assert float(torch.linalg.vector_norm(x + v * 2.0 ** -110)) <= 3e-7 * norm
