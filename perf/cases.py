"""What the performance of this library is measured on: the steps of the two-site update, each
through the call a program makes for it, and three whole calls (two ground-state searches and a
real-time step).

Sizes are those of the library's workloads (8-site chain at chi = 32; dense update at
chi = 256; 32 chains at chi = 256; U(1) bonds and gates at chi = 512) and the ranges around
them.  All tensors are complex128, as the library takes them.  Inputs are made from the seed
alone; one context serves all states, as one context serves a program."""
import math

import numpy as np
import torch

from paper_1610_02244_gb300 import synth, tnt

DEV = "cuda:0"
CDT = torch.complex128
D = 4  # Bose-Hubbard MPO bond dimension

_CTX = []


def _ctx():
    if not _CTX:
        _CTX.append(tnt.Context(0))
    return _CTX[0]


def listed():
    return [
        # the matvec of a small chain (8 sites, chi = 32): a few small launches
        {"name": "heff_fp64_chi32", "kind": "heff", "chl": 32, "chr": 32, "d": 4, "mixed": False},
        # the FP64 matvec of the dense update: every step of an FP64 solve, the FP64 finish of others
        {"name": "heff_fp64_chi256", "kind": "heff", "chl": 256, "chr": 256, "d": 4, "mixed": False},
        # the split-TF32 matvec of the same update, the bulk of a mixed-precision solve
        {"name": "heff_mixed_chi256", "kind": "heff", "chl": 256, "chr": 256, "d": 4, "mixed": True},
        # one FP64 matvec of 32 chains in lock step over their uneven charge blocks
        {"name": "heff_u1_chains32", "kind": "heff_u1", "chains": 32, "chi": 256, "d": 5, "sectors": 9},
        # an FP64 eigensolve to 1e-12, restarts and all, on a mid-sized bond
        {"name": "lanczos_fp64_chi64", "kind": "lanczos", "chl": 64, "chr": 64, "d": 4},
        # growth of the left and of the right environment by one site
        {"name": "env_chi256", "kind": "env", "chl": 256, "chr": 256, "d": 4},
        # theta from two sites and a gate on it, at the quench's bond bound
        {"name": "theta_gate_chi512", "kind": "theta_gate", "chl": 512, "chm": 512, "chr": 512, "d": 5},
        # truncated SVD of the dense update's theta (1024 x 1024 to 256)
        {"name": "svd_1024", "kind": "svd", "m": 1024, "n": 1024, "chi": 256, "right": False},
        # truncated SVD over the uneven charge blocks of a U(1) bond
        {"name": "svd_u1_chi512", "kind": "svd_u1", "chi": 512, "d": 5, "sectors": 15, "right": True},
        # the 8-site ground-state search from a random state: many small updates
        {"name": "dmrg_l8_chi32", "kind": "dmrg", "L": 8, "d": 4, "chi": 32, "sweeps": 3, "mott": False,
         "mixed": False},
        # a ground-state search from the Mott state with the bond dimension growing into chi = 128
        {"name": "dmrg_l12_chi128", "kind": "dmrg", "L": 12, "d": 4, "chi": 128, "sweeps": 3, "mott": True,
         "mixed": True},
        # one second-order Trotter step of a chain at its bond bound, with the densities after it
        {"name": "tebd_l10_chi128", "kind": "tebd", "L": 10, "d": 5, "chi": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("heff", "heff", "heff", "heff_u1", "lanczos", "env", "theta_gate", "svd", "svd", "svd_u1",
                       "dmrg", "tebd"))
    if kind == "heff":
        return {"kind": kind, "chl": _log(rng, 12, 256), "chr": _log(rng, 12, 256), "d": rng.randint(2, 4),
                "mixed": rng.random() < 0.34}
    if kind == "heff_u1":
        return {"kind": kind, "chains": _log(rng, 1, 32), "chi": _log(rng, 32, 256), "d": rng.randint(3, 5),
                "sectors": rng.randint(5, 11)}
    if kind == "lanczos":
        return {"kind": kind, "chl": _log(rng, 12, 64), "chr": _log(rng, 12, 64), "d": rng.randint(2, 4)}
    if kind == "env":
        return {"kind": kind, "chl": _log(rng, 16, 256), "chr": _log(rng, 16, 256), "d": rng.randint(2, 4)}
    if kind == "theta_gate":
        return {"kind": kind, "chl": _log(rng, 16, 512), "chm": _log(rng, 16, 512), "chr": _log(rng, 16, 512),
                "d": rng.randint(2, 5)}
    if kind == "svd":
        m, n = _log(rng, 24, 1024), _log(rng, 24, 1024)
        return {"kind": kind, "m": m, "n": n, "chi": max(4, min(m, n) // rng.randint(2, 4)),
                "right": rng.random() < 0.5}
    if kind == "svd_u1":
        return {"kind": kind, "chi": _log(rng, 48, 512), "d": rng.randint(2, 5), "sectors": rng.randint(5, 15),
                "right": rng.random() < 0.5}
    if kind == "dmrg":
        return {"kind": kind, "L": rng.randint(6, 10), "d": rng.randint(3, 4), "chi": _log(rng, 16, 96),
                "sweeps": rng.randint(2, 3), "mott": rng.random() < 0.5, "mixed": rng.random() < 0.5}
    return {"kind": kind, "L": rng.randint(6, 10), "d": rng.randint(3, 5), "chi": _log(rng, 24, 128)}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(DEV)
    g.manual_seed(seed)
    return g


def _gauss(g, *shape):
    return torch.randn(*shape, dtype=CDT, device=DEV, generator=g)


def _hermitian_env(g, chi):
    """Gaussian environment E[a', w, a] whose channels pair as the MPO's operators do."""
    h0, h3, b = _gauss(g, chi, chi), _gauss(g, chi, chi), _gauss(g, chi, chi)
    h = math.sqrt(0.5)
    return torch.stack(((h0 + h0.mH) * h, b, b.mH, (h3 + h3.mH) * h), dim=1).contiguous()


def _block_env(g, chi, side):
    """Environment of a gapped block in its eigenbasis: unit channel, levels 0 and 1..11, and a
    Gaussian boundary operator with its adjoint."""
    ident, ham = (3, 0) if side == "left" else (0, 3)
    E = torch.zeros(chi, D, chi, dtype=CDT, device=DEV)
    lam = torch.rand(chi, dtype=torch.float64, device=DEV, generator=g)
    lam = 1.0 + 10.0 * torch.sort(lam)[0]
    lam[0] = 0.0
    B = _gauss(g, chi, chi) / math.sqrt(chi)
    E[:, ident, :] = torch.eye(chi, dtype=CDT, device=DEV)
    E[:, ham, :] = torch.diag(lam).to(CDT)
    E[:, 1, :] = B
    E[:, 2, :] = B.mH
    return E


def _mpo_site(seed, d, k=0):
    """A Bose-Hubbard MPO tensor (J = 1) with its interaction drawn from the seed."""
    U = 1.0 + 7.0 * np.random.default_rng([seed, k]).random()
    return torch.from_numpy(tnt.bh_mpo_site(d - 1, 1.0, U)).to(DEV)


def _graded(g, m, n, chi):
    """Gaussian m x n matrix with singular values falling by about four decades per chi of them, as
    the Schmidt values of a two-site tensor do."""
    r = min(m, n)
    s = torch.exp(torch.arange(r, dtype=torch.float64, device=DEV) * (-math.log(1e4) / chi))
    return (_gauss(g, m, r) * s) @ _gauss(g, r, n) / math.sqrt(m * n)


def _u1_labels(c):
    return (synth.gaussian_sector_labels(c["chi"], c["sectors"], 2.0, 31),
            synth.gaussian_sector_labels(c["chi"], c["sectors"], 2.0, 33))


def _u1_blocks(c):
    """Row labels, column labels and the (charge, rows, columns) blocks of theta[(a s1), (s2 b)]."""
    qa, qb = _u1_labels(c)
    s = np.arange(c["d"])
    rq = (qa[:, None] + s[None, :]).reshape(-1)
    cq = (qb[None, :] - s[:, None]).reshape(-1)
    blocks = []
    for q in np.unique(rq):
        rows, cols = np.nonzero(rq == q)[0], np.nonzero(cq == q)[0]
        if len(rows) and len(cols):
            blocks.append((int(q), rows, cols))
    return rq, cq, blocks


def prepare(case, seed):
    c, g, ctx = case, _gen(seed), _ctx()
    kind = c["kind"]
    s = {"case": c, "ctx": ctx}
    if kind in ("heff", "lanczos"):
        env = (lambda n, side: _hermitian_env(g, n)) if kind == "heff" else (lambda n, side: _block_env(g, n, side))
        s["L"], s["R"] = env(c["chl"], "left"), env(c["chr"], "right")
        s["W1"], s["W2"] = _mpo_site(seed, c["d"]), _mpo_site(seed, c["d"], 1)
        s["theta"] = _gauss(g, c["chl"], c["d"], c["d"], c["chr"])
    elif kind == "heff_u1":
        qa, qb = _u1_labels(c)
        ma = torch.from_numpy(synth.env_mask(qa, qa)).to(DEV)
        mb = torch.from_numpy(synth.env_mask(qb, qb)).to(DEV)
        s["probs"] = [tnt.U1Problem(_hermitian_env(g, c["chi"]) * ma, _mpo_site(seed, c["d"], 2 * k),
                                    _mpo_site(seed, c["d"], 2 * k + 1), _hermitian_env(g, c["chi"]) * mb,
                                    qa, qb, synth.BH_WQ) for k in range(c["chains"])]
        s["x"] = _gauss(g, sum(ctx.u1_size(p) for p in s["probs"]))
    elif kind == "env":
        s["L"], s["R"] = _hermitian_env(g, c["chl"]), _hermitian_env(g, c["chr"])
        s["W"] = _mpo_site(seed, c["d"])
        s["A"] = _gauss(g, c["chl"], c["d"], c["chr"]) / math.sqrt(c["chl"] * c["d"])
    elif kind == "theta_gate":
        s["A"] = _gauss(g, c["chl"], c["d"], c["chm"])
        s["B"] = _gauss(g, c["chm"], c["d"], c["chr"])
        U = 1.0 + 7.0 * np.random.default_rng(seed).random()
        s["G"] = torch.from_numpy(tnt.bh_bond_gate(c["d"] - 1, 1.0, U, 0.0, 0.5, 0.5, 0.01)).to(DEV)
    elif kind == "svd":
        s["M"] = _graded(g, c["m"], c["n"], c["chi"])
    elif kind == "svd_u1":
        rq, cq, blocks = _u1_blocks(c)
        M = torch.zeros(len(rq), len(cq), dtype=CDT, device=DEV)
        for q, rows, cols in blocks:  # sector weights and spectra around the mean filling
            w = math.exp(-((q - 32.5) ** 2) / 16.0)
            b = w * _graded(g, len(rows), len(cols), max(2.0, 0.4 * min(len(rows), len(cols))))
            M[torch.from_numpy(rows).to(DEV)[:, None], torch.from_numpy(cols).to(DEV)[None, :]] = b
        s["M"], s["rq"], s["cq"] = M, rq, cq
    elif kind == "dmrg":
        s["U"] = 2.0 + 4.0 * np.random.default_rng(seed).random()
        if not c["mott"]:
            s["tensors"], s["charges"] = synth.random_charged_mps(synth.rng(seed), c["L"], c["d"], c["L"], c["chi"])
    else:  # tebd
        ctx.set_params(chi_max=c["chi"], precision=tnt.TNT_PREC_FP64)
        tensors, charges = synth.random_charged_mps(synth.rng(seed), c["L"], c["d"], c["L"], c["chi"], "gauss")
        s["mps"] = ctx.mps_create(tensors, charges, c["chi"])
        U = 1.0 + 7.0 * np.random.default_rng(seed).random()
        s["tebd"] = ctx.tebd_create(s["mps"], c["d"] - 1, 1.0, U, 0.01)
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "heff":
        return ctx.heff_apply(s["L"], s["W1"], s["W2"], s["R"], s["theta"],
                              precision=tnt.TNT_PREC_MIXED if c["mixed"] else tnt.TNT_PREC_FP64)
    if kind == "heff_u1":
        return ctx.heff_apply_u1(s["probs"], s["x"])[0]
    if kind == "lanczos":
        ctx.set_params(precision=tnt.TNT_PREC_FP64)
        x = s["theta"].clone()  # the call overwrites its start vector
        return {"E": ctx.lanczos_ground(s["L"], s["W1"], s["W2"], s["R"], x)["E"], "x": x}
    if kind == "env":
        return ctx.env_left(s["L"], s["W"], s["A"]), ctx.env_right(s["R"], s["W"], s["A"])
    if kind == "theta_gate":
        theta = ctx.theta_form(s["A"], s["B"])
        return theta, ctx.gate_apply(s["G"], theta)
    if kind in ("svd", "svd_u1"):
        # singular vectors are free up to phases: the truncated tensor U (S V^H) is what they define
        ctx.set_params(chi_max=c["chi"])
        U, X, S, bq, _ = ctx.svd_trunc(s["M"], s.get("rq"), s.get("cq"),
                                       side=tnt.TNT_SVD_RIGHT if c["right"] else tnt.TNT_SVD_LEFT)
        return {"theta": ctx.matmul(U, X), "S": S, "bond_q": bq}
    if kind == "dmrg":
        ctx.set_params(chi_max=c["chi"], precision=tnt.TNT_PREC_MIXED if c["mixed"] else tnt.TNT_PREC_FP64)
        if c["mott"]:
            mps = ctx.mps_product(synth.mott_occupations(c["L"]), c["d"], c["chi"])
        else:
            mps = ctx.mps_create(s["tensors"], s["charges"], c["chi"])
        search = ctx.dmrg_create(mps, ctx.mpo_bose_hubbard(c["L"], c["d"] - 1, 1.0, s["U"]))
        for _ in range(c["sweeps"]):
            search.sweep()
        return {"E": search.update_energies(), "density": mps.density(), "corr": mps.bdagb()}
    ctx.set_params(chi_max=c["chi"], precision=tnt.TNT_PREC_FP64)
    s["tebd"].step()
    return {"density": s["mps"].density(), "norm2": s["mps"].norm2()}


# ---------------------------------------------------------------- least work of one pass
def _heff_work(chl, chr_, d):
    n = chl * d * d * chr_
    return {"bytes": 16.0 * (D * (chl * chl + chr_ * chr_) + 2 * D * D * d * d + 2 * n),
            "flops": 8.0 * D * n * (chl + chr_)}


def _u1_heff_work(c):
    qa, qb = _u1_labels(c)
    ca = {int(q): int((qa == q).sum()) for q in np.unique(qa)}
    cb = {int(q): int((qb == q).sum()) for q in np.unique(qb)}
    wq, flops, n = synth.BH_WQ, 0.0, 0
    for q, na in ca.items():
        for s in range(2 * c["d"] - 1):  # s1 + s2, with its number of pairs
            pairs = min(s + 1, 2 * c["d"] - 1 - s)
            nb = cb.get(q + s, 0)
            n += pairs * na * nb
            flops += 8.0 * pairs * na * nb * sum(ca.get(q + w, 0) + cb.get(q + s + w, 0) for w in wq)
    env = sum(ca[q] * ca.get(q + w, 0) for q in ca for w in wq) + sum(cb[q] * cb.get(q + w, 0) for q in cb for w in wq)
    return {"bytes": 16.0 * c["chains"] * (2 * n + env), "flops": c["chains"] * flops}


def _svd_work(m, n, k):
    g = min(m, n)  # Gram product, its reduction, the projections and the product of the factors
    return 4.0 * m * n * g + 16.0 / 3.0 * g ** 3 + 16.0 * m * n * k


def work(case):
    c, kind = case, case["kind"]
    if kind == "heff":
        return _heff_work(c["chl"], c["chr"], c["d"])
    if kind == "heff_u1":
        return _u1_heff_work(c)
    if kind == "lanczos":  # a converged solve of such a bond takes about 150 matvecs
        w, n = _heff_work(c["chl"], c["chr"], c["d"]), c["chl"] * c["d"] ** 2 * c["chr"]
        return {"bytes": w["bytes"], "flops": 150.0 * (w["flops"] + 32.0 * 16 * n)}
    if kind == "env":
        site = c["chl"] * c["d"] * c["chr"]
        return {"bytes": 16.0 * (2 * site + 2 * D * (c["chl"] ** 2 + c["chr"] ** 2)),
                "flops": 16.0 * D * site * (c["chl"] + c["chr"])}
    if kind == "theta_gate":
        n = c["chl"] * c["d"] ** 2 * c["chr"]
        return {"bytes": 16.0 * (c["d"] * c["chm"] * (c["chl"] + c["chr"]) + 2 * n),
                "flops": 8.0 * n * c["chm"] + 8.0 * n * c["d"]}
    if kind == "svd":
        return {"bytes": 16.0 * (2.0 * c["m"] * c["n"] + c["chi"] * (c["m"] + c["n"])),
                "flops": _svd_work(c["m"], c["n"], c["chi"])}
    if kind == "svd_u1":
        blocks = _u1_blocks(c)[2]
        k = c["chi"] / max(1, sum(min(len(r), len(q)) for _, r, q in blocks))
        full = c["chi"] * c["d"]
        return {"bytes": 16.0 * (2.0 * full * full + 2.0 * c["chi"] * full),
                "flops": sum(_svd_work(len(r), len(q), k * min(len(r), len(q))) for _, r, q in blocks)}
    # whole calls: about 20 matvecs an update, or one truncated SVD a gate, at the bonds' sizes
    ch = [min(c["chi"], c["d"] ** min(j, c["L"] - j)) for j in range(c["L"] + 1)]
    sites = sum(ch[j] * c["d"] * ch[j + 1] for j in range(c["L"]))
    flops = 0.0
    for j in range(c["L"] - 1):
        m, n = ch[j] * c["d"], ch[j + 2] * c["d"]
        if kind == "dmrg":
            flops += 2 * c["sweeps"] * (20 * _heff_work(ch[j], ch[j + 2], c["d"])["flops"] + _svd_work(m, n, ch[j + 1]))
        else:
            flops += 1.5 * _svd_work(m, n, ch[j + 1])
    blocks = 0.2  # share of the dense work that the charge blocks leave
    return {"bytes": 2 * 16.0 * blocks * sites, "flops": blocks * flops}


# ---------------------------------------------------------------- the same in plain torch
def _heff_exact(L, W1, W2, R, x):
    t = torch.tensordot(L, x, dims=([2], [0]))                    # a' w s1 s2 b
    t = torch.einsum("awstb,wvpqst->avpqb", t, torch.einsum("wups,uvqt->wvpqst", W1, W2))
    return torch.einsum("avpqb,cvb->apqc", t, R)


def _ground_exact(s):
    """Lowest eigenpair by one long Lanczos run with full re-orthogonalisation; as in the call, the
    eigenvector's phase is that of its overlap with the start vector."""
    x0 = s["theta"]
    v = x0 / torch.linalg.norm(x0)
    V, a, b = [v.reshape(-1)], [], []
    for k in range(400):
        w = _heff_exact(s["L"], s["W1"], s["W2"], s["R"], V[-1].reshape(x0.shape)).reshape(-1)
        a.append(float(torch.vdot(V[-1], w).real))
        Q = torch.stack(V)
        for _ in range(2):
            w = w - (Q.conj() @ w) @ Q
        b.append(float(torch.linalg.norm(w)))
        if k % 10 == 9 or b[-1] < 1e-14:
            e, y = torch.linalg.eigh(torch.diag(torch.tensor(a, dtype=torch.float64)) +
                                     torch.diag(torch.tensor(b[:-1], dtype=torch.float64), 1) +
                                     torch.diag(torch.tensor(b[:-1], dtype=torch.float64), -1))
            if b[-1] * abs(float(y[-1, 0])) <= 1e-13 * abs(float(e[0])):
                break
        V.append(w / b[-1])
    x = y[:, 0].to(DEV).to(CDT) @ Q
    ov = torch.vdot(x, V[0])
    return float(e[0]), (x * (ov / ov.abs()) / torch.linalg.norm(x)).reshape(x0.shape)


def _svd_exact(M, rq, cq, chi):
    blocks = [(0, np.arange(M.shape[0]), np.arange(M.shape[1]))] if rq is None else \
        [(int(q), np.nonzero(rq == q)[0], np.nonzero(cq == q)[0]) for q in np.unique(rq)]
    M = M.cpu()
    parts, vals = [], []
    for b, (q, rows, cols) in enumerate(blocks):
        if not len(rows) or not len(cols):
            continue
        U, S, Vh = torch.linalg.svd(M[rows[:, None], cols[None, :]], full_matrices=False)
        parts.append((q, rows, cols, U, S, Vh))
        vals.append(S)
    kept = torch.sort(torch.cat(vals), descending=True)[0][:chi]
    theta, out_s, out_q = torch.zeros_like(M), [], []
    for q, rows, cols, U, S, Vh in parts:
        k = int((S >= kept[-1]).sum())
        theta[rows[:, None], cols[None, :]] = (U[:, :k] * S[:k]) @ Vh[:k]
        out_s.append(S[:k])
        out_q += [q] * k
    return {"theta": theta.to(DEV), "S": torch.cat(out_s).numpy(), "bond_q": np.array(out_q, dtype=np.int64)}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("dmrg", "tebd"):
        return None  # a truncated search or step has no closed form
    s = prepare(case, seed)
    if kind == "heff":
        return _heff_exact(s["L"], s["W1"], s["W2"], s["R"], s["theta"])
    if kind == "lanczos":
        E, x = _ground_exact(s)
        return {"E": E, "x": x}
    if kind == "heff_u1":
        qa, qb = _u1_labels(case)
        mask = torch.from_numpy(synth.theta_mask(qa, case["d"], qb)).to(DEV)
        # the labels are sorted: the compact vector is the allowed entries in dense order
        flat = torch.nonzero(mask.reshape(-1))[:, 0]
        out, at = [], 0
        for p in s["probs"]:
            th = torch.zeros(mask.numel(), dtype=CDT, device=DEV)
            th[flat] = s["x"][at:at + len(flat)]
            y = _heff_exact(*(p.tensors[k] for k in (0, 1, 2, 3)), th.reshape(mask.shape))
            out.append(y.reshape(-1)[flat])
            at += len(flat)
        return torch.cat(out)
    if kind == "env":
        t = torch.einsum("awx,xsm->awsm", s["L"], s["A"])
        t = torch.einsum("awsm,wvps->avpm", t, s["W"])
        left = torch.einsum("apn,avpm->nvm", s["A"].conj(), t)
        t = torch.einsum("asb,cvb->ascv", s["A"], s["R"])
        t = torch.einsum("ascv,wvps->awpc", t, s["W"])
        return left, torch.einsum("npc,awpc->nwa", s["A"].conj(), t)
    if kind == "theta_gate":
        theta = torch.tensordot(s["A"], s["B"], dims=([2], [0]))
        d = case["d"]
        return theta, torch.einsum("pqst,astb->apqb", s["G"].reshape(d, d, d, d), theta)
    return _svd_exact(s["M"], s.get("rq"), s.get("cq"), case["chi"])
