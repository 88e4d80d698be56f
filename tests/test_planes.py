"""The GSM path, plane by plane (csrc/plane.cuh): its identity in FP64 on the CPU, and on the GPU the
same GSM source through the plane kernels and as an uploaded CSDA through the general passes."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from gpu_cases import oracle_source, rel

D, LAM = 20e-6, 633e-9


def _planes(N, z, gsm, m, farfield):
    """W = s conj E(a') E(d') sum_{a,d} e^{+-} H(b'; a, d) T(c'; a, d), per (b', c'), in FP64."""
    n = np.arange(N) - N // 2
    dx = LAM * z / (N * D)
    q = lambda d: np.exp(1j * np.pi * (n * d) ** 2 / (LAM * z))  # noqa: E731
    sgn = (-1.0) ** np.arange(N)
    ein = np.ones(N) if farfield else q(D)
    F = (sgn * ein)[:, None] * (sgn * ein)[None, :] * m
    E = sgn * q(dx)
    x = n * D
    sS, sM, A = gsm
    G = np.exp(-(x[:, None] ** 2 + x[None, :] ** 2) / (4 * sS ** 2) - (x[:, None] - x[None, :]) ** 2 / (2 * sM ** 2))
    w = np.exp(-2j * np.pi * np.outer(np.arange(N), np.arange(N)) / N)
    H = np.einsum("k,kb,ab,bd->kad", E.conj(), w.conj(), A * F.conj(), G)
    T = np.einsum("k,kc,cd,ac->kad", E, w, F, G)
    W = np.einsum("ia,bad,cad,ld->ibcl", w.conj(), H, T, w, optimize=True)
    return (D * D / (LAM * z)) ** 2 * E.conj()[:, None, None, None] * E * W


@pytest.mark.parametrize("N,farfield,masked", [(4, False, True), (6, True, True), (8, False, False)])
def test_plane_identity(N, farfield, masked):
    rng = np.random.default_rng(N)
    m = rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N)) if masked else np.ones((N, N))
    gsm = (2.1 * D, 1.3 * D, 0.7)
    W, _ = O.propagate_fft(O.apply_mask(O.gsm_source(N, D, *gsm), m), D, LAM, 0.02, farfield=farfield)
    assert rel(_planes(N, 0.02, gsm, m, farfield), W) < 1e-12


# Each path is an FP32 DFT over 4 log2 N radix-2 levels of unit-modulus factors: a relative L2 error of at most
# 2^-24 sqrt(4 log2 N) x 3 (3.2 roundings a level and axis, in quadrature) <= 1e-6 at N = 256, so the two
# paths differ by at most 2e-6.
@pytest.mark.gpu
@pytest.mark.parametrize("N", [2, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96])
@pytest.mark.parametrize("farfield,aperture,lens,mask", [(False, False, False, True), (True, True, False, False),
                                                         (False, True, True, True)])
def test_planes_against_the_general_passes(N, farfield, aperture, lens, mask):
    import torch
    import paper_2203_02734_gb300 as pw
    gsm, z, P1 = (5 * D, 1.5 * D, 0.8), 0.3, (N // 2, N // 3)
    m = WL.to_c64(WL.phase_screen(N, seed=3)) if mask else None
    W0 = torch.from_numpy(WL.to_c64(oracle_source(N, D, LAM, gsm=gsm))).cuda()
    out = []
    for array in (False, True):
        c = pw.CSD(N, D, LAM)
        c.source_array(W0) if array else c.source_gsm(*gsm)
        if aperture:
            c.source_aperture(0.4 * N * D)
        if lens:
            c.source_lens(z)
        if mask:
            c.source_mask(torch.from_numpy(m).cuda())
        (c.propagate_farfield if farfield else c.propagate_fresnel)(z)
        out.append([t.cpu().numpy().astype(np.complex128) for t in (c.W, c.spectral_density(), c.degree_of_coherence(*P1))])
        pw.pw_csd_check(c.h)
        c.close()
    assert rel(out[0][0], out[1][0]) < 2e-6
    assert rel(out[0][1], out[1][1]) < 2e-6
    d = np.arange(N)
    M = out[0][0]
    assert np.array_equal(out[0][1].real, M[d[:, None], d[None, :], d[:, None], d[None, :]].real)
    ok = out[1][1].real >= 1e-2 * out[1][1].real.max()  # mu: 1 / sqrt(S) amplifies W's error tenfold at most
    assert np.abs(out[0][2] - out[1][2])[ok].max() < 2e-5


# The allocation-free call shares the kernel of N <= 16 (small.cuh); direct sums of N terms per axis stay
# within the bound above (2^-24 sqrt(4 N) x 3 <= 1.5e-6 at N = 16 each).
@pytest.mark.gpu
@pytest.mark.parametrize("N", [2, 4, 6, 8, 12, 16, 24])
@pytest.mark.parametrize("aperture,mask", [(False, True), (True, False)])
def test_noalloc_against_the_general_passes(N, aperture, mask):
    import torch
    import paper_2203_02734_gb300 as pw
    gsm, z = (5 * D, 1.5 * D, 0.8), 0.3
    m = torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=4))).cuda() if mask else None
    ap = 0.4 * N * D if aperture else 0.0
    W, S = torch.zeros((N,) * 4, dtype=torch.complex64, device="cuda"), torch.zeros((N, N), device="cuda")
    pw.pw_propagate_gsm_fresnel_noalloc(N, D, LAM, z, *gsm, ap, 0.0, m.data_ptr() if mask else None, W.data_ptr(),
                                        W.numel() * 8, S.data_ptr(), torch.cuda.current_stream().cuda_stream)
    c = pw.CSD(N, D, LAM)
    c.source_array(torch.from_numpy(WL.to_c64(oracle_source(N, D, LAM, gsm=gsm))).cuda())
    if aperture:
        c.source_aperture(ap)
    if mask:
        c.source_mask(m)
    c.propagate_fresnel(z)
    c128 = lambda t: t.cpu().numpy().astype(np.complex128)  # noqa: E731
    assert rel(c128(W), c128(c.W)) < 3e-6
    assert rel(c128(S), c128(c.spectral_density())) < 3e-6
    c.close()


# The direct sums of N <= 16 are as accurate as the fast transforms that they replaced, whose relative L2 error of W
# at these sizes was 1.55e-7 in the mean over sources like these; 1.65e-7 allows for the draw of the sources.
@pytest.mark.gpu
@pytest.mark.parametrize("N", [12, 16])
def test_small_planes_are_as_accurate_as_the_passes(N):
    import torch
    import paper_2203_02734_gb300 as pw
    err = []
    for seed in range(12):
        r = np.random.default_rng([N, seed])
        gsm, z = (r.uniform(4, 6) * D, r.uniform(0.7, 1.0) * D, r.uniform(0.5, 1.5)), r.uniform(0.2, 1.2)
        m = WL.to_c64(WL.phase_screen(N, seed=seed + 1))
        c = pw.CSD(N, D, LAM)
        c.source_gsm(*gsm)
        c.source_mask(torch.from_numpy(m).cuda())
        c.propagate_fresnel(z)
        W, _ = O.propagate_fft(O.apply_mask(O.gsm_source(N, D, *gsm), m.astype(complex)), D, LAM, z)
        err.append(rel(c.W.cpu().numpy().astype(complex), W))
        c.close()
    assert np.mean(err) < 1.65e-7, np.mean(err)
