"""torch.autograd on a stream that is not the handle's: inputs that the caller's stream has still to write, a
handle that is busy, and memory that the caller's stream is still reading when an output takes it over."""
import pytest

pytestmark = pytest.mark.gpu

D, LAM = 20e-6, 633e-9
BUSY = 40_000_000  # clock cycles, some 20 ms


def _model(kind, N, direct=True):
    from paper_2203_02734_gb300.autograd import CSDPropagation, GSMPropagation
    if kind == "csd":
        return CSDPropagation(N, D, LAM, 0.5, P1=(N // 2, N // 2 - 1))
    m = GSMPropagation(N, D, LAM, 0.5, P1=(N // 2, N // 2 - 1))
    m.direct = m.direct and direct
    return m


def _inputs(kind, N, torch):
    g = torch.Generator(device="cuda").manual_seed(3)
    if kind == "csd":
        u = torch.randn(N * N, 3, dtype=torch.complex64, device="cuda", generator=g)
        return (u.conj() @ u.T).reshape(N, N, N, N)
    return 0.5 + 0.5 * torch.rand(N, N, device="cuda", generator=g)


def _step(model, kind, x):
    """Outputs and gradients of one step."""
    x = x.detach().requires_grad_()
    S, mu = model(x) if kind == "csd" else model(5 * D, 1.5 * D, 1.2, x)
    (S.sum() / S.detach().max() + (mu.real ** 2).sum()).backward()
    return [S.detach(), mu.detach(), x.grad]


@pytest.mark.parametrize("kind,direct", [("gsm", True), ("gsm", False), ("csd", True)])
def test_other_stream_gives_the_same(kind, direct):
    import torch
    N = 32
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    x = _inputs(kind, N, torch)
    torch.cuda.synchronize()
    with torch.cuda.stream(a):
        model = _model(kind, N, direct)
        ref = [t.clone() for t in _step(model, kind, x)]
    torch.cuda.synchronize()
    for rep in range(3):
        with torch.cuda.stream(b):
            late = torch.zeros_like(x)
            pool = torch.full((64, N, N), 3.0, device="cuda")  # what the caller's stream still reads
        torch.cuda.synchronize()
        with torch.cuda.stream(a):
            torch.cuda._sleep(BUSY)  # the handle's stream is busy when the outputs are read
        with torch.cuda.stream(b):
            torch.cuda._sleep(2 * BUSY)
            late.copy_(x)  # the input is written behind the caller's stream
            kept = pool.sum()
            del pool
            out = [t + 0 for t in _step(model, kind, late)]
        torch.cuda.synchronize()
        assert float(kept) == 3.0 * 64 * N * N
        for r, o in zip(ref, out):
            assert torch.equal(torch.view_as_real(r) if r.is_complex() else r, torch.view_as_real(o) if o.is_complex() else o)
    model.close()


def test_capture_on_another_stream():
    import torch
    from paper_2203_02734_gb300.autograd import GSMPropagation
    N, a = 32, torch.cuda.Stream()
    x = _inputs("gsm", N, torch)
    with torch.cuda.stream(a):
        model = GSMPropagation(N, D, LAM, 0.5)
    torch.cuda.synchronize()
    with torch.no_grad():
        ref = [t.clone() for t in model(5 * D, 1.5 * D, 1.2, x)]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            out = model(5 * D, 1.5 * D, 1.2, x)
    for t in out:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    for r, o in zip(ref, out):
        assert torch.equal(torch.view_as_real(r) if r.is_complex() else r, torch.view_as_real(o) if o.is_complex() else o)
    model.close()
