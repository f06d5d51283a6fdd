"""A Lanczos solve that ends in an error leaves nothing of its own in flight: the calls after it, which
use the same scratch and pinned buffers, give what they give on a fresh context, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnt():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt as t
    return t


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


@pytest.mark.parametrize("chi,d", [(5, 2), (24, 3), (40, 4)])
def test_calls_after_a_failed_solve(tnt, chi, d):
    g = synth.rng(chi)
    L, R = dev(synth.block_env(g, chi, "left")), dev(synth.block_env(g, chi, "right"))
    W = dev(tnt.bh_mpo_site(d - 1, 1.0, 3.0))
    th = dev(synth.complex_gaussian(g, (chi, d, d, chi)))
    fresh = tnt.Context(0)
    want = fresh.heff_apply(L, W, W, R, th, precision=tnt.TNT_PREC_FP64)
    x0 = th.clone()
    e0 = fresh.lanczos_ground(L, W, W, R, x0)["E"]
    bad = L.clone()
    bad[0, 0, 1] = float("nan")
    ctx = tnt.Context(0)
    for _ in range(20):
        with pytest.raises(tnt.TntError) as e:
            ctx.lanczos_ground(bad, W, W, R, th.clone())
        assert e.value.code == 7
        assert torch.equal(ctx.heff_apply(L, W, W, R, th, precision=tnt.TNT_PREC_FP64), want)
    x = th.clone()
    assert ctx.lanczos_ground(L, W, W, R, x)["E"] == e0
    assert torch.equal(x, x0)
