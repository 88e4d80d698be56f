"""The tensor-core contractions (csrc/dense_tc.cuh) against the FP32 ones on the CUDA cores, at the sizes
where their tiling changes: Np = N rounded up to 16 around one CTA or two per tile (Np = 128 / 144), two
or three operand buffers (NOUT = 208 / 224), column counts that leave a ragged last tile, and inputs that
are only 8-byte aligned.

An accumulation of 6 Np / 16 steps whose partial sums are truncated to 24 bits is off by at most half of
that many units of 2^-23, 5e-6 at Np = 224; contractions add in quadrature, and the FP32 path's own error
is 1e-6, so the two stay within 1e-5."""
import numpy as np
import pytest

import oracle as O
import workloads as WL

pytestmark = pytest.mark.gpu

D, LAM = 20e-6, 633e-9


def _run(N, Nz, mode, source, farfield):
    import torch
    import paper_2203_02734_gb300 as pw
    c = pw.CSD(N, D, LAM)
    pw.pw_csd_set_padding(c.h, Nz)
    pw.pw_csd_set_dft_mode(c.h, mode)
    source(c, pw, torch)
    (c.propagate_farfield if farfield else c.propagate_fresnel)(0.3)
    S = c.spectral_density()
    pw.pw_csd_check(c.h)
    W = c.W
    c.close()
    return W, S


def _compare(N, Nz, source, farfield=False):
    W1, S1 = _run(N, Nz, 1, source, farfield)
    W2, S2 = _run(N, Nz, 2, source, farfield)
    # 2-norms over slabs of the first axis (the arrays are up to 15 GB)
    num = sum(float((W2[a] - W1[a]).abs().double().square().sum()) for a in range(N))
    den = sum(float(W1[a].abs().double().square().sum()) for a in range(N))
    assert (num / den) ** 0.5 < 1e-5
    assert float((S2 - S1).double().norm() / S1.double().norm()) < 1e-5


@pytest.mark.parametrize("N,Nz", [(10, 0), (16, 26), (18, 0), (34, 60), (126, 0), (130, 200), (210, 0)])
def test_gsm_with_masks(N, Nz):
    def source(c, pw, torch):
        c.source_gsm(5 * D, 1.5 * D, 0.8)
        c.source_mask(torch.from_numpy(WL.to_c64(WL.phase_screen(N, seed=4))).cuda())
        c.source_aperture(0.4 * N * D)
    _compare(N, Nz, source)


@pytest.mark.parametrize("N,offset", [(10, 0), (18, 1), (34, 1), (54, 0), (130, 1)])
@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e30])
def test_uploaded_array(N, offset, scale):
    import torch
    g = torch.Generator(device="cuda").manual_seed(N)
    buf = torch.randn(N ** 4 + 1, dtype=torch.complex64, device="cuda", generator=g)
    buf *= scale / N  # outputs of size `scale`, inside the FP32 range

    def source(c, pw, _):
        pw.pw_source_array(c.h, buf[offset:].data_ptr(), 0)
        c.source_aperture(0.45 * N * D)
    _compare(N, 0, source, farfield=True)


def test_non_finite_input_stays_in_its_propagation():
    import torch
    N = 18
    W0 = torch.randn(N, N, N, N, dtype=torch.complex64, device="cuda")
    W0[3, 4, 5, 6] = complex(float("inf"), 0.0)
    W, S = _run(N, 0, 2, lambda c, pw, _: c.source_array(W0, False), False)
    assert not bool(torch.isfinite(W).any())  # every output takes every input


# Masks that leave only the tail of the source: in the tables a and d meet the other point's mask only in the
# product (see dense_tc.cuh).  Against FP64 on sampled rows; FP32 accumulation as above, 1e-5.
@pytest.mark.parametrize("sM", [1.5, 50.0])
@pytest.mark.parametrize("N,Nz,kind", [(90, 0, "disc"), (90, 0, "opening"), (54, 80, "disc"), (136, 0, "opening")])
def test_gsm_tail_through_a_mask(N, Nz, kind, sM):
    import torch
    import paper_2203_02734_gb300 as pw
    n, sS = np.arange(N) - N // 2, N / 18
    r2 = n[:, None] ** 2 + n[None, :] ** 2
    m = (r2 >= (6.4 * sS) ** 2) if kind == "disc" else ((n[:, None] - int(8 * sS)) ** 2 + n[None, :] ** 2 <= 9)
    m = WL.to_c64(WL.phase_screen(N, seed=4) * m)
    z, rows = 0.3, [(N // 2, N // 2), (3, N - 2), (N // 3, N // 2 + 5)]
    c = pw.CSD(N, D, LAM)
    pw.pw_csd_set_padding(c.h, Nz)
    pw.pw_csd_set_dft_mode(c.h, 2)
    c.source_gsm(sS * D, sM * D, 1.0)
    c.source_mask(torch.from_numpy(m).cuda())
    c.propagate_fresnel(z)
    pw.pw_csd_check(c.h)
    ref = O.propagate_rows_gsm_padded(m.astype(complex), N, D, LAM, z, sS * D, sM * D, 1.0, rows, Nz or N)
    out = np.array([c.W[r].cpu().numpy() for r in rows]).astype(complex)
    assert np.linalg.norm(out - ref) < 1e-5 * np.linalg.norm(ref)
    c.close()
