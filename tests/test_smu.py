"""S and mu of a GSM source without its CSDA (csrc/smu.cuh): the identity in FP64 on the CPU, and on the
GPU the batch's instances without W against the same instances through the handle (plane kernels)."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from gpu_cases import rel

D, LAM = 20e-6, 633e-9


@pytest.mark.parametrize("N,farfield,P1", [(4, False, (1, 3)), (6, True, (5, 0)), (8, False, (4, 4))])
def test_correlation_identity(N, farfield, P1):
    rng = np.random.default_rng(N)
    z, (sS, sM, A) = 0.02, (2.1 * D, 1.3 * D, 0.7)
    m = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))
    W, dx = O.propagate_fft(O.apply_mask(O.gsm_source(N, D, sS, sM, A), m), D, LAM, z, farfield=farfield)
    n, L = np.arange(N) - N // 2, 2 * N
    sgn = (-1.0) ** np.arange(N)
    ein = sgn * (1 if farfield else np.exp(1j * np.pi * (n * D) ** 2 / (LAM * z)))
    E = sgn * np.exp(1j * np.pi * (n * dx) ** 2 / (LAM * z))
    h = np.exp(-(n * D) ** 2 / (4 * sS ** 2))
    k = lambda u: np.exp(-(u * D) ** 2 / (2 * sM ** 2))  # noqa: E731
    P = (ein * h)[:, None] * (ein * h)[None, :] * m
    u = np.where(np.arange(L) < N, np.arange(L), np.arange(L) - L)
    ku = np.where(u == -N, 0.0, k(u))
    Ph = np.fft.fft2(P, s=(L, L))
    C = np.fft.ifft2(np.abs(Ph) ** 2) * ku[:, None] * ku[None, :]
    C = C[:N, :N] + C[N:, :N] + C[:N, N:] + C[N:, N:]
    s = A * (D * D / (LAM * z)) ** 2
    assert rel(s * np.fft.fft2(C), O.spectral_density(W)) < 1e-12
    K = np.fft.fft(ku)
    im, jm = (2 * P1[0] - np.arange(L)) % L, (2 * P1[1] - np.arange(L)) % L
    R = np.fft.ifft2(K[:, None] * K[None, :] * Ph[im][:, jm].conj())[:N, :N]
    row = s * np.conj(E[P1[0]] * E[P1[1]]) * E[:, None] * E[None, :] * np.fft.fft2(P * R)
    assert rel(row, W[P1]) < 1e-12


# Both sides are FP32 FFTs with a relative L2 error below 1e-6 (see test_planes.py); S and the row of mu
# then differ by at most 2e-6 in L2, and mu where S >= 1e-2 max S by ten times that.
@pytest.mark.gpu
@pytest.mark.parametrize("N,n,pool,mask", [(16, 40, 1, True), (16, 3, 2, False), (32, 5, 1, True), (64, 2, 1, True),
                                           (96, 2, 1, False), (128, 2, 1, True)])
def test_batch_without_w_matches_the_handle(N, n, pool, mask):
    import torch
    import paper_2203_02734_gb300 as pw
    m = torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=7))).cuda() if mask else None
    S = torch.full((n, N, N), float("nan"), device="cuda")
    mu = torch.full((n, N, N), float("nan"), dtype=torch.complex64, device="cuda")
    insts, P1 = [], [(0, N - 1), (N // 2, N // 3), (N - 1, 2)]
    for i in range(n):
        q = pw.pw_instance()
        q.N, q.dxi_m, q.lambda_m, q.z_m, q.farfield = N, D, LAM * (1 + 0.01 * i), 0.3 + 0.05 * i, i % 2
        q.sigma_S_m, q.sigma_mu_m, q.amplitude = 5 * D, 1.5 * D, 0.8 + 0.1 * i
        q.aperture_m, q.lens_f_m = (0.4 * N * D, 0.4) if i % 3 == 1 else (0.0, 0.0)
        q.dev_mask = m.data_ptr() if mask else 0
        (q.iP, q.jP), q.dev_S, q.dev_mu = P1[i % 3], S[i].data_ptr(), mu[i].data_ptr()
        insts.append(q)
    nb = pw.pw_batch_workspace_bytes(insts, pool)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    b = pw.pw_batch_create(insts, pool, ws.data_ptr(), nb, torch.cuda.current_stream().cuda_stream)
    pw.pw_batch_run(b)
    pw.pw_batch_check(b)
    pw.pw_batch_destroy(b)
    for i in {0, 1, n - 1}:
        q = insts[i]
        c = pw.CSD(N, D, q.lambda_m)
        c.source_gsm(q.sigma_S_m, q.sigma_mu_m, q.amplitude)
        if q.aperture_m:
            c.source_aperture(q.aperture_m)
            c.source_lens(q.lens_f_m)
        if mask:
            c.source_mask(m)
        (c.propagate_farfield if q.farfield else c.propagate_fresnel)(q.z_m)
        Sh = c.spectral_density().cpu().numpy().astype(np.float64)
        muh = c.degree_of_coherence(q.iP, q.jP).cpu().numpy().astype(np.complex128)
        c.close()
        Sb, mub = S[i].cpu().numpy().astype(np.float64), mu[i].cpu().numpy().astype(np.complex128)
        assert rel(Sb, Sh) < 2e-6
        sp = Sh[q.iP, q.jP]
        if sp >= 1e-2 * Sh.max():
            ok = Sh >= 1e-2 * Sh.max()
            assert np.abs(mub - muh)[ok].max() < 2e-5


# The handle's call against the propagation it stands for, at every grid size with a plan; bounds as above.
@pytest.mark.gpu
@pytest.mark.parametrize("N", [4, 6, 8, 12, 24, 48, 96, 128])
@pytest.mark.parametrize("farfield", [False, True])
def test_handle_s_mu_matches_the_propagation(N, farfield):
    import torch
    import paper_2203_02734_gb300 as pw
    m = torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=9))).cuda()
    P1 = (N // 2 - 1, N // 2)
    c = pw.CSD(N, D, LAM)
    c.source_gsm(5 * D, 1.5 * D, 1.3)
    c.source_mask(m)
    c.source_aperture(0.45 * N * D)
    c.source_lens(0.6)
    S = torch.empty(N, N, device="cuda")
    mu = torch.empty(N, N, dtype=torch.complex64, device="cuda")
    pw.pw_gsm_s_mu(c.h, 0.3, farfield, *P1, S.data_ptr(), mu.data_ptr())
    assert abs(c.sampling() / D - 1) < 1e-12  # the current plane is untouched
    (c.propagate_farfield if farfield else c.propagate_fresnel)(0.3)
    Sp, mup = c.spectral_density(), c.degree_of_coherence(*P1)
    with pytest.raises(pw.PwError, match="PW_ESTATE"):
        pw.pw_gsm_s_mu(c.h, 0.3, farfield, *P1, S.data_ptr(), mu.data_ptr())
    c.close()
    Sp, S = Sp.cpu().numpy().astype(np.float64), S.cpu().numpy().astype(np.float64)
    assert rel(S, Sp) < 2e-6
    ok = Sp >= 1e-2 * Sp.max()
    if ok[P1]:
        assert np.abs((mu - mup).cpu().numpy()[ok]).max() < 2e-5
