"""An MPO tensor with a NaN or an infinity gives a non-finite result, and a Lanczos solve with it the
error for one, also where the entry only meets zeros of the other tensor."""
import numpy as np
import pytest
import torch

from oracle import bose_hubbard as bh
from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("which", [0, 1])
def test_non_finite_entry_beside_zeros(bad, which):
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    ctx = tnt.Context(0)
    dev = lambda x: torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")  # noqa: E731
    g = synth.rng(4)
    chi, d = 12, 3
    Ws, _, _ = bh.bh_mpo(4, d - 1, 1.0, 2.0)
    W = [Ws[1].copy(), Ws[2].copy()]
    W[1 - which][1, :] = 0.0
    W[1 - which][:, 1] = 0.0
    W[which][1 if which else 0, 0 if which else 1, 0, 0] = bad
    L, R = dev(synth.hermitian_env(g, chi)), dev(synth.hermitian_env(g, chi))
    th = dev(synth.complex_gaussian(g, (chi, d, d, chi)))
    y = ctx.heff_apply(L, dev(W[0]), dev(W[1]), R, th, precision=tnt.TNT_PREC_FP64)
    assert not torch.isfinite(torch.view_as_real(y)).all()
    with pytest.raises(tnt.TntError) as e:
        ctx.lanczos_ground(L, dev(W[0]), dev(W[1]), R, th)
    assert e.value.code == 7
