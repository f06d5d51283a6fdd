"""Where there is no device memory for the slices of FP64 products, the products run on the FP64 units
instead of failing, and give those units' bits: a caller's allocator that grants what the FP64
units' engine asked for, and no more."""
import numpy as np
import pytest
import torch

from oracle import bose_hubbard as bh
from paper_1610_02244_gb300 import synth
from test_gpu_u1 import dev, problem, u1_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnt():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt as t
    return t


class Limited:
    """A context whose allocator records its largest request and refuses those above a limit."""

    def __init__(self, tnt, engine, limit=None):
        alloc0, free0 = tnt.torch_allocator(0, torch.cuda.current_stream(0))
        self.largest, self.refused = 0, 0

        def alloc(n):
            if limit is not None and n > limit:
                self.refused += 1
                raise MemoryError
            self.largest = max(self.largest, n)
            return alloc0(n)
        self.ctx = tnt.Context(0, allocator=(alloc, free0))
        self.ctx.set_fp64_gemm(engine)


def both(tnt, call):
    """The FP64 units' result, and the default engine's where only their memory is to be had."""
    a = Limited(tnt, tnt.TNT_FP64_GEMM_FMA)
    want = call(a.ctx)
    b = Limited(tnt, tnt.TNT_FP64_GEMM_TC, max(a.largest, 1 << 16))
    got = call(b.ctx)
    return want, got, b.refused


def test_products(tnt):
    g = synth.rng(1)
    A, B = dev(synth.complex_gaussian(g, (500, 200))), dev(synth.complex_gaussian(g, (200, 700)))
    want, got, refused = both(tnt, lambda c: c.matmul(A, B))
    assert refused > 0 and torch.equal(want, got)
    # the same context works on afterwards
    L, R = dev(synth.hermitian_env(g, 96)), dev(synth.hermitian_env(g, 96))
    Ws, _, _ = bh.bh_mpo(4, 3, 1.0, 2.0)
    th = dev(synth.complex_gaussian(g, (96, 4, 4, 96)))
    want, got, refused = both(tnt, lambda c: c.heff_apply(L, dev(Ws[1]), dev(Ws[2]), R, th))
    assert torch.equal(want, got)


def test_block_sparse_matvec(tnt):
    qa, qb = synth.gaussian_sector_labels(192, 9, 2.0, 15), synth.gaussian_sector_labels(200, 9, 2.0, 17)
    Le, W1, W2, Re, th = u1_inputs(5, qa, qb, 4)
    p = problem(Le, W1, W2, Re, qa, qb)
    x = tnt.Context(0).u1_pack(p, dev(th))
    want, got, refused = both(tnt, lambda c: c.heff_apply_u1([p], x)[0])
    assert refused > 0 and torch.equal(want, got)
