"""The early end of the SVD's reduction where many rows are of the largest one's size: a matrix that
falls into a flat diagonal part, empty rows and one small value behind them, given without
labels.  The reduction meets an empty row first, and only the trace that is really left says
that the value behind it counts.  With 920 candidates of 1200 the last row is none of the
candidates that an end at the empty row would keep.

The value's square is 1500 to 4000 eps of the largest row's (above the 1000 eps that the
eigensolver splits off).  Diagonal matrices reduce exactly, so the value comes out to rounding."""
import numpy as np
import pytest
import torch

from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    c = tnt.Context(0)
    c.set_params(chi_max=920)
    return c


@pytest.mark.parametrize("eigenvalue", [1500, 4000])
@pytest.mark.parametrize("seed", range(12))
def test_small_value_behind_empty_rows(ctx, seed, eigenvalue):
    n, r = 1200, 900
    g = synth.rng(seed)
    s = np.zeros(n)
    s[:r] = g.uniform(0.9, 1.0, r)
    s[0] = 1.0
    s[n - 1] = np.sqrt(eigenvalue * 2.0 ** -52)
    M = np.diag(s.astype(np.complex128))
    S = np.sort(ctx.svd_trunc(torch.from_numpy(M).to("cuda:0"), side=seed % 2)[2])[::-1]
    assert len(S) == r + 1
    assert np.abs(S[:r] - np.sort(s)[::-1][:r]).max() <= 1e-13
    assert abs(S[r] / s[n - 1] - 1.0) <= 1e-10
