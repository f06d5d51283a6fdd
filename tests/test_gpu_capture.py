"""theta = A B under stream capture (`tnt_theta_form`: device output only, no synchronisation): a first
call inside a capture works whatever engine its size takes outside, and a captured product
keeps its slice buffer when later calls need a larger one."""
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


@pytest.mark.parametrize("warm", [False, True])
@pytest.mark.parametrize("chl,chm,chr_,d", [(64, 80, 96, 3), (48, 180, 33, 4)])
def test_theta_in_a_capture(tnt, warm, chl, chm, chr_, d):
    stream = torch.cuda.Stream()
    ctx = tnt.Context(0, stream=stream)
    A, B = rand(1, chl, d, chm), rand(2, chm, d, chr_)  # on slices outside a capture
    out = torch.zeros(chl, d, d, chr_, dtype=torch.complex128, device="cuda:0")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        sliced = ctx.theta_form(A, B).clone() if warm else None
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_FMA)
    with torch.cuda.stream(stream):
        fma = ctx.theta_form(A, B).clone()
    ctx.set_fp64_gemm(tnt.TNT_FP64_GEMM_TC)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        ctx.theta_form(A, B, out=out)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, sliced if warm else fma)
    # a larger product makes the slice buffer grow; the graph still owns the old one
    big = ctx.theta_form(rand(3, 300, 4, 400), rand(4, 400, 4, 300))
    A.copy_(rand(5, chl, d, chm))
    torch.cuda.synchronize()
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    ref = np.tensordot(A.cpu().numpy(), B.cpu().numpy(), axes=([2], [0]))
    assert np.abs(out.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
    assert torch.isfinite(torch.view_as_real(big)).all()
