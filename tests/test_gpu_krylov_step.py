"""One FP64 Krylov step's kernels where they can go wrong: the fused Gram-Schmidt step at
vector lengths around its slices (fewer elements than SMs, ragged last CTA, basis kept in
shared memory or not) and the lowest pair of T_k at the lengths around a warp's two rows per
lane, against dense numpy diagonalisation of the same H_eff.

Tolerances: the solve stops at a residual of 1e-12 |E|, so E is exact to rounding (1e-12) and
the vector to 1e-12 |E| / gap; with the gap of at least 0.05 |E| of these operators that is
2e-11, taken as 1e-9."""
import numpy as np
import pytest
import torch

from oracle import bose_hubbard as bh
from oracle import contract as oc
from paper_1610_02244_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    return tnt.Context(0)


def dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to("cuda:0")


def dense_heff(Le, W1, W2, Re, shape):
    n = int(np.prod(shape))
    cols = [oc.heff_apply(Le, W1, W2, Re, e.reshape(shape)).reshape(-1) for e in np.eye(n, dtype=np.complex128)]
    return np.array(cols).T


@pytest.mark.parametrize("chl,chr_,d,cap", [(1, 2, 2, 8), (3, 5, 2, 32), (7, 9, 3, 33), (8, 10, 3, 64), (9, 13, 3, 31),
                                            (6, 5, 4, 2), (16, 17, 2, 3)])
def test_solve_against_dense(ctx, chl, chr_, d, cap):
    g = synth.rng(100 * chl + chr_)
    Le, Re = synth.block_env(g, chl, "left"), synth.block_env(g, chr_, "right")
    Ws, _, _ = bh.bh_mpo(4, d - 1, 1.0, 2.0)
    th = synth.complex_gaussian(g, (chl, d, d, chr_))
    H = dense_heff(Le, Ws[1], Ws[2], Re, th.shape)
    ev, vec = np.linalg.eigh((H + H.conj().T) / 2)
    old = ctx.params()
    ctx.set_params(krylov_cap=cap, lanczos_maxit=300)
    try:
        x = dev(th)
        r = ctx.lanczos_ground(dev(Le), dev(Ws[1]), dev(Ws[2]), dev(Re), x)
    finally:
        ctx.set_params(krylov_cap=old["krylov_cap"], lanczos_maxit=old["lanczos_maxit"])
    x = x.cpu().numpy().reshape(-1)
    if r["converged"]:
        assert abs(r["E"] - ev[0]) <= 1e-12 * abs(ev[0]) + 1e-12
        assert 1.0 - abs(np.vdot(vec[:, 0], x)) <= 1e-9
    else:  # a cap of two or three vectors restarts slowly: the quotient still bounds from above
        assert cap <= 3 and ev[0] - 1e-12 <= r["E"] <= ev[-1]
    assert abs(np.linalg.norm(x) - 1.0) <= 1e-12
    assert abs(np.vdot(x, H @ x).real - r["E"]) <= 1e-11 * max(1.0, abs(ev).max())


@pytest.mark.parametrize("chl,chr_,d", [(19, 2, 2), (64, 38, 2), (120, 111, 2), (150, 150, 2), (129, 130, 4)])
def test_basis_stays_orthonormal(ctx, chl, chr_, d):
    """Lengths below, at and above one element per SM, with the basis slice inside and outside
    shared memory: the Rayleigh quotient of the returned vector equals the reported energy, as
    it does only for an orthonormal basis."""
    g = synth.rng(chl + 7 * chr_)
    Le, Re = synth.block_env(g, chl, "left"), synth.block_env(g, chr_, "right")
    Ws, _, _ = bh.bh_mpo(4, d - 1, 1.0, 2.0)
    W = Ws[1:3]
    th = synth.complex_gaussian(g, (chl, d, d, chr_))
    x = dev(th)
    r = ctx.lanczos_ground(dev(Le), dev(W[0]), dev(W[1]), dev(Re), x)
    y = oc.heff_apply(Le, W[0], W[1], Re, x.cpu().numpy().reshape(th.shape)).reshape(-1)
    xn = x.cpu().numpy().reshape(-1)
    assert r["converged"] == 1
    assert abs(np.linalg.norm(xn) - 1.0) <= 1e-12
    assert abs(np.vdot(xn, y).real - r["E"]) <= 1e-11 * max(1.0, abs(r["E"]))
    assert np.linalg.norm(y - r["E"] * xn) <= 1e-9 * max(1.0, abs(r["E"]))
