"""The truncated SVD's block-parallel eigen path (`csrc/heig.cu`) where it can go wrong: blocks
around the sizes at which a CTA group, a panel of reflectors or a route changes, many
uneven blocks in one call, and exactly low-rank blocks, whose reduction leaves trailing
matrices that shrink by sixteen decades per column.

Tolerances: the Gram matrix and its reduction resolve singular values to about
n eps sigma_max in absolute terms (1e-13 with room for n up to 600), U (or V) is orthonormal to
the Newton-Schulz steps' 1e-13.  The factors multiply back to M up to what the kept vectors
miss of its range: a Gram matrix larger than the rank mixes the smallest kept direction with
its null space by an angle of n eps (sigma_max / sigma_k)^2, which moves M by that times
sigma_k."""
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
    return tnt.Context(0)


def check(ctx, M, rq=None, cq=None, side=0):
    U, X, S, bq, info = ctx.svd_trunc(torch.from_numpy(np.ascontiguousarray(M)).to("cuda:0"), rq, cq, side=side)
    U, X = U.cpu().numpy(), X.cpu().numpy()
    assert np.all(np.isfinite(U)) and np.all(np.isfinite(X)) and np.all(np.isfinite(S))
    sref = np.linalg.svd(M, compute_uv=False)
    k = len(S)
    assert np.abs(np.sort(S)[::-1] - sref[:k]).max() <= 1e-13 * sref[0]
    assert np.linalg.norm(sref[k:]) <= 2e-8 * sref[0]  # the default truncation error
    Q = U if side == 0 else X.conj().T
    assert np.abs(Q.conj().T @ Q - np.eye(k)).max() <= 1e-13
    null = len(sref) * 2.0 ** -52 * sref[0] ** 2 / S.min()
    assert np.linalg.norm(U @ X - M) <= np.linalg.norm(sref[k:]) + 1e-13 * len(sref) * sref[0] + null


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 64, 65, 127, 129, 192, 193, 257, 320, 600])
@pytest.mark.parametrize("side", [0, 1])
def test_single_block(ctx, n, side):
    g = synth.rng(n)
    check(ctx, synth.complex_gaussian(g, (n, n + 5)) @ np.diag(np.logspace(0, -3, n + 5)), side=side)


@pytest.mark.parametrize("m,n,rank", [(20, 1, 1), (20, 2, 2), (64, 3, 2), (200, 40, 1), (250, 250, 5)])
@pytest.mark.parametrize("side", [0, 1])
def test_exactly_low_rank(ctx, m, n, rank, side):
    for seed in range(12):
        g = synth.rng(1000 * rank + seed)
        if seed % 2:  # small integers: exact cancellations
            M = (g.integers(-3, 4, (m, rank)) + 1j * g.integers(-3, 4, (m, rank))) @ g.integers(-3, 4, (rank, n))
            M[0, 0] += 1
        else:
            M = synth.complex_gaussian(g, (m, rank)) @ synth.complex_gaussian(g, (rank, n))
        check(ctx, M.astype(np.complex128), side=side)


@pytest.mark.parametrize("sizes", [(500, 400, 300, 200, 100, 50, 20, 5, 1), (7,) * 60, (260, 255, 1, 193, 192)])
@pytest.mark.parametrize("side", [0, 1])
def test_many_uneven_blocks(ctx, sizes, side):
    g = synth.rng(sum(sizes))
    rq = np.concatenate([np.full(s, i) for i, s in enumerate(sizes)])
    cq = np.concatenate([np.full(max(1, s - i % 3), i) for i, s in enumerate(sizes)])
    M = synth.complex_gaussian(g, (len(rq), len(cq))) * (rq[:, None] == cq[None, :])
    M *= np.logspace(0, -2, len(cq))[None, :]
    check(ctx, M, rq, cq, side=side)


@pytest.mark.parametrize("n", [3, 33, 130, 400])
@pytest.mark.parametrize("spectrum", ["graded", "equal", "exact_pairs", "near_pairs", "two_levels"])
def test_spacings_of_the_eigenvalues(ctx, n, spectrum):
    """Brackets that hold one eigenvalue, several or a whole cluster: the determinants at their
    ends guide the bisection in the first case only."""
    h = np.linspace(1.0, 0.3, (n + 1) // 2)
    s = {"graded": np.logspace(0, -4, n), "equal": np.ones(n), "exact_pairs": np.repeat(h, 2)[:n],
         "near_pairs": (np.repeat(h, 2) * np.tile([1.0, 1.0 - 1e-9], h.size))[:n],
         "two_levels": np.where(np.arange(n) < n // 2, 1.0, 1e-3)}[spectrum]
    g = synth.rng(n)
    U, V = (np.linalg.qr(synth.complex_gaussian(g, (n, n)))[0] for _ in range(2))
    check(ctx, (U * s) @ V)


@pytest.mark.parametrize("total", [1, 255, 256, 257, 513, 4096, 4099])
def test_selection_at_its_thread_counts(ctx, total):
    """The global order and the truncation error over as many candidates as one, a thread's four,
    or all of its eight hold.  Blocks of eight neighbouring values (1 to 1e-9 over all): the
    Gram matrix of a block resolves them to 8 eps (largest / smallest)^2 < 1e-13 relative, and sums
    of their squares over all to 1e-10 with room."""
    s = np.logspace(0, -9, total)
    g = synth.rng(total)
    lab = np.arange(total) // 8
    M = np.zeros((total, total), dtype=np.complex128)
    for q in range(lab[-1] + 1):
        i = np.flatnonzero(lab == q)
        U, V = (np.linalg.qr(synth.complex_gaussian(g, (i.size, i.size)))[0] for _ in range(2))
        M[np.ix_(i, i)] = (U * s[i]) @ V
    perm = g.permutation(lab[-1] + 1)  # charges in another order than the values
    order = np.argsort(perm[lab], kind="stable")
    M, q = M[np.ix_(order, order)], perm[lab][order]
    U, X, S, bq, info = ctx.svd_trunc(torch.from_numpy(M).to("cuda:0"), q, q)
    tail = np.append(np.cumsum((s ** 2)[::-1])[::-1], 0.0) / (s ** 2).sum()  # discards from index i on
    chi = max(1, int(np.argmax(np.sqrt(tail) < 1e-8)))  # the default 2-norm error
    assert info["chi"] == chi == len(S)
    assert np.abs(np.sort(S)[::-1] / s[:chi] - 1.0).max() <= 1e-12
    assert abs(info["err"] - np.sqrt(tail[chi])) <= 1e-10 * np.sqrt(tail[chi])
    assert np.array_equal(np.sort(bq), np.sort(perm[lab[:chi]]))
