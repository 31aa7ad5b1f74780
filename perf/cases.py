"""The measured work of this framework: what a user's program has it do, through the public Python
entry points (TNMC, TNMCPeriodic, TNMCServer), from one small pilot up to a filled GPU.

A case is a dict of plain values with a "kind":
  pass      a context that serves batch after batch: new realizations (couplings on the device), the
            environments with log Z, n proposals per chain, Metropolis, observables
  point     the same for one point of an acceptance sweep: the context is made and closed in the call
  propose   more proposals from environments that are in hand, with their spins
  evaluate  log q and the conditionals of given configurations, environments in hand
  torus     steps of the periodic chains (every step builds the environments of every region)
  serve     a stream of mixed requests through the request server, until all have answered
"""
import math

import numpy as np
import torch

import paper_2409_06538_gb300 as tn

OBS_FLOAT = ("E", "E2", "m_abs", "m2", "m4", "q", "q_abs", "q2", "q4", "m_edge", "m_edge_abs", "m_edge2")
OBS_INT = ("n_prop", "n_acc", "n_meas", "n_meas_q", "clamps", "n_tests", "status")


def _case(kind, L, chi, R, n, precision="tf32", p=0.109, chains=2, compression="canonical", **more):
    return dict(kind=kind, L=L, chi=chi, R=R, n=n, precision=precision, p=p, chains=chains, compression=compression,
                **more)


def listed():
    return [
        # the pilot that picks a bond dimension for one (L, p): a few tiny realizations, where the
        # launches, the context and the synchronisations are what is paid for
        dict(_case("point", 8, 4, 8, 100, p=0.10926), name="pilot_l8_chi4"),
        # one point of the acceptance sweep at a small lattice; chi below what the tensor cores take
        dict(_case("point", 16, 8, 64, 200, p=0.10926), name="sweep_l16_chi8"),
        # the exactness check: nothing truncated, 100 realizations x 1000 proposals, all in FP64
        dict(_case("pass", 8, 16, 100, 500, "fp64", 0.10), name="exact_l8_chi16_fp64"),
        # the FP64 path where it truncates: the parity reference of every other path
        dict(_case("pass", 24, 16, 32, 100, "fp64"), name="batch_l24_chi16_fp64"),
        # a thousand realizations in one launch, 2000 proposals each: disorder averages at L = 32
        dict(_case("pass", 32, 16, 1024, 1000), name="batch_l32_chi16"),
        # as many chi = 32 realizations as the SMs hold builds of, 500 proposals each; the lattice
        # size is what a pass of a second allows
        dict(_case("pass", 48, 32, 448, 250), name="batch_l48_chi32"),
        # the batch that the throughput is quoted on (64 realizations x 2 chains x 250), at L = 64: the
        # build leaves most of the GPU idle and is what the latency of a batch consists of
        dict(_case("pass", 64, 32, 64, 250), name="batch_l64_chi32"),
        # the cheaper compression on the same kind of batch
        dict(_case("pass", 48, 32, 64, 100, compression="zipup"), name="zipup_l48_chi32"),
        # the widest bond dimension, few realizations
        dict(_case("pass", 20, 64, 8, 100), name="wide_l20_chi64"),
        # long chains: thousands of proposals from environments that are already built
        dict(_case("propose", 64, 32, 64, 500), name="propose_l64_chi32"),
        # likelihoods of given configurations; odd lattice side, bond dimension between the tiles' sizes
        dict(_case("evaluate", 33, 12, 24, 200), name="evaluate_l33_chi12"),
        # periodic boundaries: one build per proposal, with the pinned lines as external fields
        dict(_case("torus", 20, 16, 32, 3), name="torus_l20_chi16"),
    ]


# microseconds of a site step of the environment build of one realization, by padded bond dimension
# (FP64: times ten), and realizations an SM builds at a time: only to keep drawn cases affordable
_STEP_US = {4: 25.0, 8: 45.0, 16: 90.0, 32: 250.0, 64: 1300.0}
_PER_SM = {4: 3, 8: 3, 16: 3, 32: 2, 64: 1}


def _pad(chi):
    return next(c for c in (4, 8, 16, 32, 64) if chi <= c)


def _seconds(c):
    """A rough time of one build and of the proposals of a case."""
    C, f64 = _pad(c["chi"]), c["precision"] == "fp64"
    R = c["R"] * (c["chains"] if c["kind"] == "torus" else 1)
    waves = math.ceil(R / (152 * (1 if f64 else _PER_SM[C])))
    build = c["L"] * (c["L"] - 1) * _STEP_US[C] * 1e-6 * waves * (10 if f64 else 1)
    spins = float(c["L"]) ** 2 * c["n"] * R * (c["chains"] if c["kind"] in ("pass", "point", "propose") else 1)
    if c["kind"] == "torus":
        return build * c["n"]
    return build + spins * C / 16 / (6e7 if f64 else 8e8 if C == 64 else 1.5e9)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(("pass", "pass", "pass", "point", "propose", "evaluate", "torus", "serve"))
        L = _log(rng, 6, 64)
        precision = rng.choice(("tf32", "tf32", "tf32", "tf32", "fp32", "bf16", "fp64"))
        if L > 20 and precision == "bf16":          # BF16 environments lose the conditionals beyond this
            precision = "tf32"
        chi = rng.choice((2, 4, 5, 8, 12, 16, 16, 24, 32, 32, 48, 64))
        if precision == "fp64":
            chi = min(chi, 32)
        R = _log(rng, 1, 512)
        n = _log(rng, 10, 1000)
        if kind == "torus":
            R, n = min(R, 64), rng.randint(1, 4)
        compression = "zipup" if kind == "pass" and rng.random() < 0.2 else "canonical"
        c = _case(kind, L, chi, R, n, precision, round(rng.uniform(0.09, 0.13), 5), 2, compression)
        if kind == "pass" and rng.random() < 0.15:
            c["fields"] = True
        if kind == "serve":
            c.update(L=min(L, 32), R=min(R, 48), n=max(n, 100), precision="tf32")
        # no drawn case costs more than about the largest listed ones, nor more memory for its spins
        if _seconds(c) < 0.6 and L * L * n * R * 2 < 4e8:
            return c


def _inputs(case, seed):
    """Realization seeds and +-J couplings (on the GPU), and the inverse temperature."""
    base = 1 + seed * 100_003
    seeds = np.arange(base, base + case["R"], dtype=np.uint64)
    beta = tn.nishimori_beta(case["p"])
    make = tn.torus_couplings_pmj if case["kind"] == "torus" else tn.couplings_pmj
    return seeds, make(case["L"], seeds, case["p"]), beta


def _context(case, J, beta, seeds):
    return tn.TNMC(case["L"], J, beta, seeds, case["chi"], precision=case["precision"], n_chains=case["chains"],
                   compression=case["compression"])


def _configurations(case, seed):
    """Configurations to be judged: states of a uniform sign with independent flips, as a chain far from
    and near to order has them."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    shape = (case["R"], case["n"], case["L"], case["L"])
    share = torch.rand(shape[:2], generator=g, device="cuda")[..., None, None] * 0.5
    return torch.where(torch.rand(shape, generator=g, device="cuda") < share, -1, 1).to(torch.int8)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        rng = np.random.default_rng(seed)
        sides = [max(4, case["L"] // 2), case["L"]]
        reqs = []
        for k in range(case["R"]):
            L = int(rng.choice(sides))
            p = float(rng.uniform(0.09, 0.13))
            reqs.append((int(seed) * 100_003 + k, L, min(case["chi"], 2 ** (L // 2)), p, tn.nishimori_beta(p),
                         int(rng.integers(100, case["n"] + 1))))
        srv = tn.TNMCServer(case["precision"], case["chains"], max_batch=32, max_inflight=4, linger_us=500,
                            mem_budget=16 << 30)
        return dict(case=case, srv=srv, reqs=reqs)
    seeds, J, beta = _inputs(case, seed)
    s = dict(case=case, seeds=seeds, J=J, beta=beta)
    if kind == "torus":
        s["ctx"] = tn.TNMCPeriodic(case["L"], J, beta, seeds, case["chi"], precision=case["precision"],
                                   n_chains=case["chains"])
    elif kind != "point":
        s["ctx"] = _context(case, J, beta, seeds)
        if case.get("fields"):
            k = np.random.default_rng(seed).integers(-1, 2, (case["R"], case["L"], case["L"]))
            s["ctx"].set_fields(k.astype(np.int8))
        if kind in ("propose", "evaluate"):
            s["ctx"].build_env(return_logz=False)
        if kind == "evaluate":
            s["spins"] = _configurations(case, seed)
    return s


def _means(obs):
    return (np.array([[o[k] for k in OBS_FLOAT] for o in obs]),
            np.array([[o[k] for k in OBS_INT] for o in obs], dtype=np.int64))


def _batch(ctx, n):
    log_z = ctx.build_env()
    out = ctx.propose(n, 0)
    flags = ctx.accept(flags=True)["flags"]
    means, counts = _means(ctx.observables(allow_numeric=True))
    return dict(log_z=log_z, logq=out["logq"], energy=out["energy"], magnet=out["magnet"], accepted=flags,
                means=means, counts=counts)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "pass":
        s["ctx"].set_couplings(s["J"], s["beta"], s["seeds"])
        return _batch(s["ctx"], case["n"])
    if kind == "point":
        ctx = _context(case, s["J"], s["beta"], s["seeds"])
        out = _batch(ctx, case["n"])
        ctx.close()
        return out
    if kind == "propose":
        out = s["ctx"].propose(case["n"], 0)
        return dict(logq=out["logq"], energy=out["energy"], magnet=out["magnet"], spins=s["ctx"].spins())
    if kind == "evaluate":
        logq, qplus = s["ctx"].eval_conditionals(s["spins"])
        return dict(logq=logq, qplus=qplus)
    if kind == "torus":
        s["ctx"].step(case["n"], 0)
        means, counts = _means(s["ctx"].observables())
        return dict(spins=s["ctx"].spins(), means=means, counts=counts)
    ids = [s["srv"].submit(*r) for r in s["reqs"]]
    got = [s["srv"].wait(i) for i in ids]
    means, counts = _means(got)
    return dict(log_z=np.array([g["log_z"] for g in got]), means=means, counts=counts)


def _site_flops(k):
    """Truncating a site of the MPO x MPS product at bond dimension k: product, QR, SVD, carried rest."""
    return 175.0 * k ** 3


def work(case):
    """Couplings and fields read, the environments written and read once, what a proposal returns
    written once; flops of the compression of every site and of the two sweeps of every proposal."""
    kind, chains, n = case["kind"], case["chains"], case["n"]
    shapes = [(case["L"], case["chi"], case["R"])]
    if kind == "serve":
        shapes = [(L, min(case["chi"], 2 ** (L // 2)), case["R"] / 2) for L in (max(4, case["L"] // 2), case["L"])]
    el = {"fp64": 8, "bf16": 2}.get(case["precision"], 4)
    nbytes = flops = 0.0
    for L, chi, R in shapes:
        items = R * (chains if kind not in ("evaluate", "torus") else 1) * n
        builds, per_build = (R, 1) if kind not in ("propose", "evaluate") else (0, 0)
        if kind == "torus":
            L, items, builds, per_build = L - 1, R * chains * n * 2, R * chains * n, 1
        # bond dimensions of a row: grown from both ends, cut at chi; the rows below the last grow too
        sites = sum(min(chi, 2.0 ** min(c, L - c, 40), 2.0 ** min(L - 1 - r, 40)) ** 3 for r in range(L - 1)
                    for c in range(1, L))
        tiles = sum(2 * min(chi, 2.0 ** min(c, L - c, 40), 2.0 ** min(L - 1 - r, 40)) ** 2 for r in range(L)
                    for c in range(1, L))
        flops += builds * per_build * _site_flops(1) * sites + items * 8.0 * tiles / 2
        nbytes += R * 2 * L * (L - 1) + builds * tiles * el + R * tiles * el * (1 if kind != "torus" else chains * n)
        nbytes += items * (16 + L * L / 8)
        if kind == "evaluate":
            nbytes += items * L * L * 9
        if kind == "propose":
            nbytes += items * L * L
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------------------------------
# The same quantities in FP64 with plain numpy, realizations as a leading batch axis.  Site tensors are
# (R, left, 2, right); index 0 of a spin is +1.
# ---------------------------------------------------------------------------------------------------

_S = np.array([1.0, -1.0])


def _absorb(row, beta, jv, jh, k):
    """One row of the network applied to the row state below it."""
    out = []
    for c, B in enumerate(row):
        R, l, _, r = B.shape
        W = np.exp(beta * jv[:, c, None, None] * np.multiply.outer(_S, _S))            # (R, x, y)
        if k is not None:
            W = W * np.exp(beta * k[:, c, None, None] * _S)
        if c == 0:
            A = W[:, None]                                                              # (R, a, x, y)
        else:
            A = W[:, None] * np.exp(beta * jh[:, c - 1, None, None] * np.multiply.outer(_S, _S))[:, :, None, :]
        T = A[:, :, None, :, :, None] * B[:, None, :, None, :, :]                       # R a l x y r
        if c == len(row) - 1:
            T = T.sum(axis=4, keepdims=True)
        out.append(T.reshape(R, T.shape[1] * l, 2, T.shape[4] * r))
    return out


def _unit(T):
    n = np.sqrt((T.reshape(len(T), -1) ** 2).sum(1))
    return T / n.reshape(-1, *([1] * (T.ndim - 1))), np.log(n)


def _truncate(A, chi, canonical):
    """Cut the bonds from the right, keeping the chi largest singular values at each; canonical: after
    a sweep of QR decompositions from the left."""
    A, logs = list(A), 0.0
    R = len(A[0])
    if canonical:
        for c in range(len(A) - 1):
            _, l, _, r = A[c].shape
            q, t = np.linalg.qr(A[c].reshape(R, l * 2, r))
            t, ln = _unit(t)
            logs = logs + ln
            A[c] = q.reshape(R, l, 2, -1)
            A[c + 1] = np.einsum("Rab,Rbxc->Raxc", t, A[c + 1], optimize=True)
    for c in range(len(A) - 1, 0, -1):
        _, l, _, r = A[c].shape
        u, sv, vt = np.linalg.svd(A[c].reshape(R, l, 2 * r), full_matrices=False)
        k = min(chi, sv.shape[1])
        A[c] = vt[:, :k].reshape(R, k, 2, r)
        rest, ln = _unit(np.einsum("Raxb,Rbk->Raxk", A[c - 1], u[:, :, :k] * sv[:, None, :k], optimize=True))
        A[c - 1] = rest
        logs = logs + ln
    A[0], ln = _unit(A[0])
    return A, logs + ln


def _flip(row):
    return [B.transpose(0, 3, 2, 1) for B in reversed(row)]


def _environments(jh, jv, beta, chi, k, zipup):
    R, L = len(jh), jh.shape[1]
    rows = [None] * L
    rows[L - 1] = [np.ones((R, 1, 2, 1))] * L
    logz = np.zeros(R)
    for r in range(L - 2, -1, -1):
        kr = None if k is None else k[:, r + 1]
        if zipup and (L - 2 - r) % 2 == 0:
            A = _absorb(_flip(rows[r + 1]), beta, jv[:, r, ::-1], jh[:, r + 1, ::-1], None if kr is None else kr[:, ::-1])
            row, ln = _truncate(A, chi, False)
            rows[r] = _flip(row)
        else:
            rows[r], ln = _truncate(_absorb(rows[r + 1], beta, jv[:, r], jh[:, r + 1], kr), chi, not zipup)
        logz = logz + ln
    h = (lambda c: np.ones((R, 2))) if k is None else (lambda c: np.exp(beta * k[:, 0, c, None] * _S))
    v = rows[0][0][:, 0] * h(0)[:, :, None]
    for c in range(1, L):
        W = np.exp(beta * jh[:, 0, c - 1, None, None] * np.multiply.outer(_S, _S))
        v = np.einsum("Rpa,Rpx,Raxb->Rxb", v, W, rows[0][c], optimize=True) * h(c)[:, :, None]
        v, ln = _unit(v)
        logz = logz + ln
    return rows, logz + np.log(v.sum(axis=(1, 2)))


def _judge(rows, jh, jv, beta, spins):
    """log q and q(+) of given configurations (R, n, L, L)."""
    R, n, L, _ = spins.shape
    qplus = np.zeros(spins.shape)
    for r in range(L):
        h = beta * jv[:, r - 1, None, :] * spins[:, :, r - 1] if r else np.zeros((R, n, L))
        right, v = np.ones((R, n, 2, 1)), [None] * L
        for c in range(L - 1, -1, -1):
            v[c] = np.matmul(right.transpose(0, 2, 1, 3), rows[r][c].transpose(0, 2, 3, 1)).transpose(0, 2, 1, 3)
            if c:
                W = np.exp(beta * jh[:, r, c - 1, None, None, None] * np.multiply.outer(_S, _S) + h[:, :, c, None, None] * _S)
                right = np.matmul(W, v[c])
                right = right / np.abs(right).max(axis=(2, 3), keepdims=True)
        left = np.ones((R, n, 1))
        for c in range(L):
            e = h[:, :, c, None] * _S
            if c:
                e = e + beta * jh[:, r, c - 1, None, None] * spins[:, :, r, c - 1, None] * _S
            w = np.maximum(np.exp(e) * (left[:, :, None, :] * v[c]).sum(-1), 0.0)
            qplus[:, :, r, c] = w[..., 0] / w.sum(-1)
            both = [np.matmul(left, rows[r][c][:, :, y]) for y in (0, 1)]
            left = np.where(spins[:, :, r, c, None] == 1, both[0], both[1])
            left = left / np.abs(left).max(axis=2, keepdims=True)
    q = np.where(spins == 1, qplus, 1.0 - qplus)
    return np.log(q).sum(axis=(2, 3)), qplus


def exact(case, seed):
    """log Z (and log q, q(+) of given configurations); draws have no 64-bit value on the FP32 paths, and
    none is attempted where the decompositions would take more than about fifteen seconds."""
    kind, L, R, C = case["kind"], case["L"], case["R"], min(case["chi"], 32)
    cost = R * L * L * (3e-5 + 3e-8 * (2 * C) ** 2.6)
    if kind in ("torus", "serve", "propose") or case["chi"] > 32 or cost > 12 or (kind == "evaluate" and R * case["n"] * L * L * C * C > 4e10):
        return None
    seeds, J, beta = _inputs(case, seed)
    J = J.cpu().numpy().astype(np.float64)
    nh = L * (L - 1)
    jh, jv = J[:, :nh].reshape(R, L, L - 1), J[:, nh:].reshape(R, L - 1, L)
    k = None
    if case.get("fields"):
        k = np.random.default_rng(seed).integers(-1, 2, (R, L, L)).astype(np.float64)
    rows, logz = _environments(jh, jv, beta, case["chi"], k, case["compression"] == "zipup")
    if kind == "evaluate":
        spins = _configurations(case, seed).cpu().numpy().astype(np.float64)
        logq, qplus = _judge(rows, jh, jv, beta, spins)
        return dict(logq=logq, qplus=qplus)
    return dict(log_z=logz, logq=None, energy=None, magnet=None, accepted=None, means=None, counts=None)
