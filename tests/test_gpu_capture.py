"""Products under stream capture (`tnt_matmul`, `tnt_theta_form`: device outputs only, no
synchronisation): a first call inside a capture works whatever engine its size takes outside,
a captured product keeps its slice buffer when later calls need a larger one, and replays
give the bits of a plain call with the same engine or, on the FP64 units, the same to rounding."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnt():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt as t
    return t


def rand(seed, *shape):
    g = torch.Generator("cuda:0")
    g.manual_seed(seed)
    return torch.randn(*shape, dtype=torch.complex128, device="cuda:0", generator=g)


def capture(stream, fn):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        fn()
    return graph


@pytest.mark.parametrize("warm", [False, True])
def test_matmul_in_a_capture(tnt, warm):
    stream = torch.cuda.Stream()
    ctx = tnt.Context(0, stream=stream)
    A, B = rand(1, 256, 128), rand(2, 128, 512)  # on slices outside a capture
    C = torch.zeros(256, 512, dtype=torch.complex128, device="cuda:0")
    torch.cuda.synchronize()
    want = ctx.matmul(A, B).clone() if warm else None
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_FMA)
    fma = ctx.matmul(A, B).clone()  # (the FP64 kernel is loaded before the capture)
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_TC)
    torch.cuda.synchronize()
    graph = capture(stream, lambda: ctx.matmul(A, B, out=C))
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(C, want if warm else fma)
    # a larger product makes the slice buffer grow; the graph still owns the old one
    big = ctx.matmul(rand(3, 1500, 700), rand(4, 700, 1300))
    A.copy_(rand(5, 256, 128))
    torch.cuda.synchronize()
    C.zero_()
    graph.replay()
    torch.cuda.synchronize()
    ref = (A.cpu().numpy() @ B.cpu().numpy())
    assert np.abs(C.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    assert torch.isfinite(torch.view_as_real(big)).all()


def test_theta_in_a_capture(tnt):
    stream = torch.cuda.Stream()
    ctx = tnt.Context(0, stream=stream)
    A, B = rand(6, 64, 3, 80), rand(7, 80, 3, 96)
    out = torch.zeros(64, 3, 3, 96, dtype=torch.complex128, device="cuda:0")
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_FMA)
    ctx.theta_form(A, B)
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_TC)
    torch.cuda.synchronize()
    graph = capture(stream, lambda: ctx.theta_form(A, B, out=out))
    graph.replay()
    torch.cuda.synchronize()
    ref = np.tensordot(A.cpu().numpy(), B.cpu().numpy(), axes=([2], [0]))
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
