"""Truncated SVD at the ends of the routes of its reduction: blocks of 1216 rows, the most that 152
CTAs hold in shared memory, and of 1217, alone and together, with a cut inside the spectrum.

Tolerances as in the block tests: singular values to 1e-13 sigma_max, the orthonormal factor to
1e-13, the product to what the cut leaves and n 1e-13 sigma_max."""
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
    c.set_params(chi_max=24)
    return c


@pytest.mark.parametrize("sizes,side", [((1216,), 0), ((1217,), 1), ((1217, 1216), 0)])
def test_largest_blocks_of_either_route(ctx, sizes, side):
    g = synth.rng(sum(sizes))
    lab = np.concatenate([np.full(n, i) for i, n in enumerate(sizes)])
    M = np.zeros((len(lab), len(lab)), dtype=np.complex128)
    for i, n in enumerate(sizes):
        r = 40
        U, V = (np.linalg.qr(synth.complex_gaussian(g, (n, r)))[0] for _ in range(2))
        b = (U * (np.logspace(0, -2, r) * (1.0 - 0.01 * i))) @ V.conj().T
        M[np.ix_(lab == i, lab == i)] = b
    s = np.sort(np.concatenate([np.logspace(0, -2, 40) * (1.0 - 0.01 * i) for i in range(len(sizes))]))[::-1]
    U, X, S, bq, info = ctx.svd_trunc(torch.from_numpy(M).to("cuda:0"), lab, lab, side=side)
    U, X = U.cpu().numpy(), X.cpu().numpy()
    assert len(S) == 24 and np.abs(np.sort(S)[::-1] - s[:24]).max() <= 1e-13
    Q = U if side == 0 else X.conj().T
    assert np.abs(Q.conj().T @ Q - np.eye(24)).max() <= 1e-13
    assert np.linalg.norm(U @ X - M) <= np.linalg.norm(s[24:]) + 1e-13 * len(lab)
