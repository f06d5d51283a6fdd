"""Small FP64 products over tiles 16, 8 and 4 rows high, the block-sparse matvec through the
slice products and through the FP64 engine, and operators with complex entries.

Bounds.  A complex part is a sum of 2 K products in any order: |error| <= (2 K + 8) 2^-53 times
the same sum over absolute values.  H_eff: the two engines each stay within 1e-12 of max|y| (K of
about 1e3 terms), so they differ by 2e-12 at most; split TF32 2e-5."""
import numpy as np
import pytest
import torch

from oracle import contract as oc
from paper_1610_02244_gb300 import synth
from test_gpu_u1 import LABELS, dev, problem, rel, u1_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1610_02244_gb300 import build as b
    b.build()
    from paper_1610_02244_gb300 import tnt
    return tnt.Context(0)


# 16 x 16 tiles: 1, 2, 6 (4 rows), 45 (8), 100 (4), 144 (16), 169 (4), 306 (16)
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (3, 17, 15), (5, 33, 17), (7, 81, 100), (65, 130, 31), (150, 150, 16),
                                   (190, 190, 17), (201, 199, 33), (281, 271, 49)])
@pytest.mark.parametrize("conj,cols", [(False, False), (True, True)])
def test_tile_heights(ctx, M, N, K, conj, cols):
    g = synth.rng(M + 5 * N + 11 * K)
    A, B = synth.complex_gaussian(g, (M, K)), synth.complex_gaussian(g, (K, N))
    Ad, Bd = (dev(A.T).T, dev(B.T).T) if cols else (dev(A), dev(B))
    ctx.set_fp64_gemm(0)
    C = ctx.matmul(Ad, Bd, conj_a=conj, conj_b=conj).cpu().numpy()
    ctx.set_fp64_gemm(1)
    ld = np.longdouble
    s = -1 if conj else 1
    Ar, Ai, Br, Bi = A.real.astype(ld), s * A.imag.astype(ld), B.real.astype(ld), s * B.imag.astype(ld)
    eps = (2 * K + 8) * 2.0 ** -53
    assert np.all(np.abs(C.real - (Ar @ Br - Ai @ Bi)) <= eps * (abs(Ar) @ abs(Br) + abs(Ai) @ abs(Bi)))
    assert np.all(np.abs(C.imag - (Ar @ Bi + Ai @ Br)) <= eps * (abs(Ar) @ abs(Bi) + abs(Ai) @ abs(Br)))


def complex_entries(g, W):
    return W * np.exp(2j * np.pi * g.random(W.shape))


@pytest.mark.parametrize("name", ["gaps", "one_sector", "gauss96", "gauss_cfg3_profile"])
@pytest.mark.parametrize("cplx", [False, True])
def test_block_sparse_engines_agree(ctx, name, cplx):
    """Structures on both sides of the line where the slice products take over."""
    qa, qb, d = LABELS[name]
    Le, W1, W2, Re, th = u1_inputs(13, qa, qb, d)
    if cplx:
        W1, W2 = complex_entries(synth.rng(1), W1), complex_entries(synth.rng(2), W2)
    p = problem(Le, W1, W2, Re, qa, qb)
    x = ctx.u1_pack(p, dev(th))
    ref = oc.heff_apply(Le, W1, W2, Re, th)
    got = []
    for engine in (1, 0):
        ctx.set_fp64_gemm(engine)
        y, _ = ctx.heff_apply_u1([p], x)
        got.append(ctx.u1_unpack(p, y).cpu().numpy())
        assert rel(got[-1], ref) < 1e-12
    ctx.set_fp64_gemm(1)
    assert rel(got[0], got[1]) < 2e-12
    y, _ = ctx.heff_apply_u1([p], x, precision=1)
    assert rel(ctx.u1_unpack(p, y).cpu().numpy(), ref) < 2e-5


@pytest.mark.parametrize("chl,chr_,d", [(5, 7, 2), (33, 40, 3), (64, 64, 3)])
@pytest.mark.parametrize("precision", [0, 1])
def test_complex_operator(ctx, chl, chr_, d, precision):
    g = synth.rng(chl + d)
    Le, Re = (synth.complex_gaussian(g, (c, 4, c)) for c in (chl, chr_))
    W1, W2 = (synth.complex_gaussian(g, (4, 4, d, d)) for _ in range(2))
    th = synth.complex_gaussian(g, (chl, d, d, chr_))
    y = ctx.heff_apply(dev(Le), dev(W1), dev(W2), dev(Re), dev(th), precision=precision).cpu().numpy()
    assert rel(y, oc.heff_apply(Le, W1, W2, Re, th)) < (1e-12, 2e-5)[precision]
