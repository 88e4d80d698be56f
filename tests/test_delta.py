"""Delta-correlated sources in closed form (csrc/delta.cuh): the identity in FP64 on the CPU, and on the GPU
the same diagonal as a recorded source and as an uploaded N^4 array through the general passes."""
import numpy as np
import pytest

import oracle as O
import workloads as WL
from gpu_cases import rel

D, LAM = 20e-6, 633e-9


@pytest.mark.parametrize("N,farfield", [(4, False), (6, True), (8, False)])
def test_difference_identity(N, farfield):
    rng = np.random.default_rng(N)
    d, z = rng.uniform(0, 1, (N, N)), 0.02
    W0 = np.zeros((N,) * 4, complex)
    i, j = np.meshgrid(np.arange(N), np.arange(N), indexing="ij")
    W0[i, j, i, j] = d
    W, dx = O.propagate_fft(W0, D, LAM, z, farfield=farfield)
    n = np.arange(N) - N // 2
    e = (-1.0) ** np.arange(N) * np.exp(1j * np.pi * (n * dx) ** 2 / (LAM * z))
    e2 = e[:, None] * e[None, :]
    Dh = np.fft.ifft2(d) * N * N
    u, v = (i[:, :, None, None] - i) % N, (j[:, :, None, None] - j) % N
    assert rel((D * D / (LAM * z)) ** 2 * e2.conj()[:, :, None, None] * e2 * Dh[u, v], W) < 1e-12


# The general passes err by at most 1e-6 (see test_planes.py), the closed form's tables less: 2e-6 apart.
@pytest.mark.gpu
@pytest.mark.parametrize("N", [2, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96])
@pytest.mark.parametrize("farfield,masked", [(False, True), (True, False)])
def test_diagonal_against_the_general_passes(N, farfield, masked):
    import torch
    import paper_2203_02734_gb300 as pw
    g = torch.Generator(device="cuda").manual_seed(N)
    d = torch.rand(N, N, device="cuda", generator=g) - 0.2
    W0 = torch.zeros(N * N, N * N, dtype=torch.complex64, device="cuda")
    W0.diagonal().copy_(0.7 * d.reshape(-1))
    m = torch.from_numpy(WL.to_c64(WL.amplitude_mask(N, seed=2))).cuda()
    out = []
    for array in (False, True):
        c = pw.CSD(N, D, LAM)
        c.source_array(W0.reshape(N, N, N, N)) if array else pw.pw_source_diagonal(c.h, d.data_ptr(), 0.7)
        if masked:
            c.source_mask(m)
            c.source_aperture(0.45 * N * D)
            c.source_lens(0.4)
        (c.propagate_farfield if farfield else c.propagate_fresnel)(0.3)
        out.append([t.cpu().numpy().astype(np.complex128) for t in (c.W, c.spectral_density())])
        c.close()
    assert rel(out[0][0], out[1][0]) < 2e-6
    assert rel(out[0][1], out[1][1]) < 2e-6


# A strong source behind weak masks: 2^120 behind 2^-70 is 2^-20 behind 1 (powers of two round nothing).
@pytest.mark.gpu
@pytest.mark.parametrize("N", [16, 96])
def test_range_of_weight_and_mask(N):
    import torch
    import paper_2203_02734_gb300 as pw
    d = torch.rand(N, N, device="cuda", generator=torch.Generator(device="cuda").manual_seed(N))
    m = torch.from_numpy(WL.to_c64(WL.amplitude_mask(N, seed=2))).cuda()
    out = []
    for A, w in [(2.0 ** -20, 1.0), (2.0 ** 120, 2.0 ** -70)]:
        c = pw.CSD(N, D, LAM)
        pw.pw_source_diagonal(c.h, d.data_ptr(), A)
        c.source_mask(m * w)
        c.propagate_fresnel(0.3)
        out.append((c.W, c.spectral_density()))
        c.close()
    for x, y in zip(*out):
        assert float(torch.linalg.vector_norm(x - y)) <= 3e-7 * float(torch.linalg.vector_norm(x))
