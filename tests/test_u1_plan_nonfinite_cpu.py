"""An MPO tensor with a NaN or an infinity reaches the grouped operator whatever zeros it meets: the
plan's W1.W2 takes the non-zero entries only where all are finite.  Host replay, no GPU."""
import numpy as np
import pytest

from oracle import bose_hubbard as bh
from paper_1610_02244_gb300 import synth
from test_u1_plan_host_cpu import replay, run_replay  # noqa: F401 (replay: a fixture)

pytestmark = pytest.mark.cpu


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("which", [0, 1])
def test_non_finite_entry_beside_zeros(replay, tmp_path, bad, which):  # noqa: F811
    g = synth.rng(3)
    qa, qb = np.array([0, 0, 1, 1, 2]), np.array([1, 2, 2, 3, 3])
    Ws, _, _ = bh.bh_mpo(4, 2, 1.0, 2.0)
    W = [Ws[1].copy(), Ws[2].copy()]
    W[1 - which][1, :] = 0.0  # bond channel 1 carries nothing in the other tensor
    W[1 - which][:, 1] = 0.0
    W[which][1 if which else 0, 0 if which else 1, 0, 0] = bad
    L = synth.hermitian_env(g, len(qa)) * synth.env_mask(qa, qa)
    R = synth.hermitian_env(g, len(qb)) * synth.env_mask(qb, qb)
    th = synth.complex_gaussian(g, (len(qa), 3, 3, len(qb))) * synth.theta_mask(qa, 3, qb)
    y, _ = run_replay(replay, tmp_path, [(qa, qb, synth.BH_WQ, L, W[0], W[1], R, th)])
    assert not np.all(np.isfinite(y))
