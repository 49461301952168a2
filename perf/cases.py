"""The workloads this library is measured on, through its public entry points.

Each case is a dict of plain values.  Its ``kind`` says which entry point it calls:

* ``decode``  -- ``QCCode.decode``: Algorithm 1 on a batch of frames (sum-product with FP32 or FP16
  messages, integer min-sum, learned min-sum), with a fixed iteration count or early stop;
* ``sparse``  -- the same for a general code given by its index tables (``SparseCode.decode``);
* ``sim``     -- ``QCCode.ber_sim``: the Monte-Carlo simulation (channel, decoding, error counts);
* ``ldpccc``  -- ``LDPCCC.window``: the pipelined decoder of the LDPC convolutional codes, pipeline full;
* ``batch``   -- ``ldpc_batch_decode``: many codes with uneven frame counts in one call;
* ``train``   -- ``ldpc_noms_forward`` + ``ldpc_noms_backward``: one training step of the learned min-sum;
* ``encode``  -- ``QCCode.encode`` + ``QCCode.channel_codewords``: random codewords sent over the channel.

Inputs are channel LLRs of the all-zero codeword over BPSK/AWGN (a consistent Gaussian N(m, 2m)),
drawn with torch from the seed.  ``exact`` restates every computed output in 64 bits with plain torch.
"""
import functools
import math
import random

import numpy as np
import torch

import paper_1204_0334_gb300 as pkg

CLIP = 30.0
ALGO = {"sp": pkg.ALGO_SP, "ms": pkg.ALGO_MS, "noms": pkg.ALGO_NOMS}
MSG = {"f32": pkg.MSG_F32, "f16": pkg.MSG_F16, "i8": pkg.MSG_I8}


def listed():
    return [
        # the parity workload and the smallest call: one package of a (3,6) code of n = 384, 30 iterations
        # (what a receiver with one short frame group at a time runs: launches and latency)
        dict(name="decode_n384_32frames", kind="decode", J=3, L=6, p=64, zero=0, gamma=32, algo="sp", msg="f32",
             iters=30, early=False, post=True, ebn0=2.0, typ=30),
        # an irregular code (zero blocks) of odd circulant size, a ragged batch, early stop, every output
        dict(name="decode_n2532_ragged", kind="decode", J=4, L=12, p=211, zero=6, gamma=1000, algo="sp", msg="f32",
             iters=30, early=True, post=True, ebn0=3.25, typ=9),
        # the long code with few frames in hand: a receiver's latency
        dict(name="decode_n18360_40frames", kind="decode", J=4, L=24, p=765, zero=0, gamma=40, algo="sp", msg="f32",
             iters=30, early=True, post=True, ebn0=3.5, typ=7),
        # the long code at throughput, the paper's fixed 30 iterations, in its waterfall (posteriors and decisions)
        dict(name="decode_n18360_2048frames", kind="decode", J=4, L=24, p=765, zero=0, gamma=2048, algo="sp",
             msg="f32", iters=30, early=False, post=True, ebn0=3.1, typ=30),
        # integer min-sum with early stop, the fixed-point receiver
        dict(name="decode_n15168_minsum", kind="decode", J=4, L=24, p=632, zero=0, gamma=4096, algo="ms", msg="i8",
             iters=30, early=True, post=False, ebn0=4.0, typ=6),
        # the Monte-Carlo simulation of the long code, FP32 messages: the benchmark's headline workload
        dict(name="sim_n18360_f32", kind="sim", J=4, L=24, p=765, gamma=4096, frames=32768, algo="sp", msg="f32",
             iters=30, ebn0=3.5, typ=7),
        # the same with FP16 message storage
        dict(name="sim_n18360_f16", kind="sim", J=4, L=24, p=765, gamma=4096, frames=32768, algo="sp", msg="f16",
             iters=30, ebn0=3.5, typ=7),
        # a general (not quasi-cyclic) irregular code through its index tables
        dict(name="sparse_n6000", kind="sparse", N=6000, M=2000, gamma=1024, algo="sp", msg="f32", iters=20,
             early=False, post=True, ebn0=2.0, typ=20),
        # continuous decoding of 1024 convolutional-code streams, 30 processors, 32 time slots a call
        dict(name="ldpccc_3x6_p128", kind="ldpccc", J=3, L=6, p=128, I=30, streams=1024, T=32, tanner=False,
             ebn0=1.5, post=True),
        # sixteen codes of different length, rate and frame count in one call, FP16 messages, early stop
        dict(name="batch_16codes_f16", kind="batch", codes=16, pmax=765, fmax=1024, msg="f16", algo="sp", iters=30,
             ebn0=3.0, draw=4, typ=12),
        # one training step of the learned min-sum on the long code, FP16 saved messages
        dict(name="train_n18360_f16", kind="train", J=4, L=24, p=765, frames=1024, T=10, ckpt=2, msg="f16",
             ebn0=3.5),
        # random codewords made and sent on the device (the transmitter's side of the simulation)
        dict(name="encode_n18360", kind="encode", J=4, L=24, p=765, gamma=4096, ebn0=3.5),
    ]


SHAPES = [(3, 6), (4, 8), (3, 9), (4, 12), (3, 12), (4, 16), (3, 18), (4, 24)]
# Eb/N0 (dB) at which a frame of this rate needs about a third of its iterations
WATERFALL = {0.5: 2.25, 2 / 3: 2.75, 0.75: 3.1, 5 / 6: 3.5}


def _ebn0(J, L, rng):
    R = 1 - J / L
    return round(min(WATERFALL.items(), key=lambda kv: abs(kv[0] - R))[1] + rng.uniform(-0.25, 0.5), 3)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["decode"] * 5 + ["sim"] * 2 + ["sparse", "ldpccc", "batch", "train", "encode"])
    if kind == "sparse":
        N = _log(rng, 200, 12000)
        M = max(40, N // rng.choice([2, 3, 4]))
        algo, msg = rng.choice([("sp", "f32"), ("sp", "f32"), ("sp", "f16"), ("ms", "i8")])
        gamma = max(1, min(4096, _log(rng, 1, 24_000_000 // N)))
        it = rng.randint(5, 30)
        return dict(kind=kind, N=N, M=M, gamma=gamma, algo=algo, msg=msg, iters=it, early=rng.random() < 0.5,
                    post=rng.random() < 0.5, ebn0=round(rng.uniform(2.25, 3.5), 3), typ=it)
    if kind == "ldpccc":
        J, L = rng.choice([(3, 6), (4, 8), (3, 9), (4, 24)])
        I = rng.randint(5, 30)
        p = _log(rng, 16, 422)
        # the decoder's store, 128 bytes per edge and 32 streams, stays within that of the listed case
        streams = max(1, min(1024, int(3.0e6 * rng.uniform(0.2, 1.0) * 32 / (J * L * p * I))))
        return dict(kind=kind, J=J, L=L, p=p, I=I, streams=streams, T=rng.randint(4, 32), tanner=rng.random() < 0.3,
                    ebn0=_ebn0(J, L, rng), post=rng.random() < 0.5)
    if kind == "batch":
        algo, msg = rng.choice([("sp", "f16"), ("sp", "f32"), ("ms", "i8")])
        it = rng.randint(10, 30)
        return dict(kind=kind, codes=rng.randint(2, 16), pmax=_log(rng, 64, 765), fmax=_log(rng, 16, 1024), msg=msg,
                    algo=algo, iters=it, ebn0=round(rng.uniform(2.75, 3.5), 3), draw=rng.randint(0, 999), typ=it // 2)
    J, L = rng.choice(SHAPES)
    p = _log(rng, 32, 765)
    N = L * p
    if kind == "train":
        frames = max(1, min(1024, _log(rng, 16, 18_000_000 // N)))
        return dict(kind=kind, J=J, L=L, p=p, frames=frames, T=rng.randint(2, 10), ckpt=rng.randint(1, 4),
                    msg=rng.choice(["f16", "f16", "f32"]), ebn0=_ebn0(J, L, rng))
    if kind == "encode":
        return dict(kind=kind, J=J, L=L, p=p, gamma=max(1, min(4096, _log(rng, 1, 75_000_000 // N))),
                    ebn0=_ebn0(J, L, rng))
    algo, msg = rng.choice([("sp", "f32"), ("sp", "f32"), ("sp", "f16"), ("ms", "i8"), ("noms", "f16")])
    it = rng.randint(10, 30)
    if kind == "sim":
        gamma = _log(rng, 64, 4096)
        return dict(kind=kind, J=J, L=L, p=p, gamma=gamma, frames=min(32768, gamma * rng.randint(2, 8)), algo=algo,
                    msg=msg, iters=it, ebn0=_ebn0(J, L, rng), typ=it // 3)
    gamma = max(1, min(4096, _log(rng, 1, 37_000_000 // N)))
    return dict(kind=kind, J=J, L=L, p=p, zero=rng.choice([0, 0, L // 3]), gamma=gamma, algo=algo, msg=msg, iters=it,
                early=rng.random() < 0.6, post=rng.random() < 0.5, ebn0=_ebn0(J, L, rng), typ=it)


# ------------------------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=256)
def _shifts(J, L, p, zero, seed):
    """A J x L shift table (-1: zero block), uniform in [0, p), redrawn while an entry closes a 4-cycle."""
    rng = np.random.default_rng([J, L, p, zero, seed, 1204])
    a = np.full((J, L), -1, dtype=np.int32)
    for j in range(J):
        for l in range(L):
            for _ in range(32):
                x = int(rng.integers(0, p))
                d = (x - a[j, :l][None, :] + a[:j, :l] - a[:j, l][:, None]) % p
                if not (d == 0).any():
                    break
            a[j, l] = x
    # at most one zero block per column, and the rows share them
    for q, l in enumerate(rng.choice(L, size=zero, replace=False) if zero else []):
        a[q % J, l] = -1
    return a


@functools.lru_cache(maxsize=16)
def _random_rows(N, M, seed):
    """(row_ptr, col_idx) of an irregular code: column degrees 2, 3, 3, 4 or 6, rows filled evenly."""
    rng = np.random.default_rng([N, M, seed, 1205])
    deg = rng.choice([2, 3, 3, 4, 6], size=N)
    while deg.sum() > 30 * M:  # rows hold at most 32 edges
        deg[rng.integers(0, N)] = 2
    stubs = np.repeat(np.arange(N), deg)
    E = len(stubs)
    rng.shuffle(stubs)
    row = np.arange(E) % M
    for _ in range(200):  # an edge drawn twice swaps its check with a random edge's
        key = row.astype(np.int64) * N + stubs
        _, first = np.unique(key, return_index=True)
        dup = np.setdiff1d(np.arange(E), first)
        if not len(dup):
            break
        other = rng.integers(0, E, size=len(dup))
        for x, y in zip(dup, other):
            row[x], row[y] = row[y], row[x]
    key = np.unique(row.astype(np.int64) * N + stubs)
    rows, cols = key // N, key % N
    ptr = np.zeros(M + 1, dtype=np.int32)
    np.add.at(ptr, rows + 1, 1)
    return np.cumsum(ptr).astype(np.int32), cols.astype(np.int32)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _llr(shape, ebn0, rate, seed):
    m = 4.0 * rate * 10.0 ** (ebn0 / 10.0)
    x = torch.randn(shape, generator=_gen(seed), device="cuda")
    return x.mul_(math.sqrt(2.0 * m)).add_(m)


def _params(T, ncirc, seed):
    """(w, o) of the learned min-sum around what training finds."""
    x = torch.rand((T, ncirc, 2), generator=_gen(seed), device="cuda")
    x[..., 0].mul_(0.2).add_(0.7)
    x[..., 1].mul_(0.2)
    return x


def _members(case):
    """(J, L, p, frames) of the codes of a mixed batch."""
    rng = np.random.default_rng([case["codes"], case["draw"], 1206])
    out = []
    for _ in range(case["codes"]):
        J, L = SHAPES[int(rng.integers(0, len(SHAPES)))]
        p = int(math.exp(rng.uniform(math.log(32), math.log(case["pmax"]))))
        out.append((J, L, min(p, 18360 // L), int(math.exp(rng.uniform(0.0, math.log(case["fmax"]))))))
    return out


def prepare(case, seed):
    k = case["kind"]
    if k == "sparse":
        rp, col = _random_rows(case["N"], case["M"], 1)
        return dict(case=case, code=pkg.SparseCode(rp, col, case["N"]),
                    llr=_llr((case["gamma"], case["N"]), case["ebn0"], 1 - case["M"] / case["N"], seed))
    if k == "batch":
        members = _members(case)
        codes = [pkg.QCCode(_shifts(J, L, p, 0, i), p) for i, (J, L, p, _) in enumerate(members)]
        counts = [g for *_, g in members]
        opts = pkg.default_opts(max_iter=case["iters"], early_stop=1, algo=ALGO[case["algo"]], msg=MSG[case["msg"]])
        s = dict(case=case, codes=codes, counts=counts, batch=_Batch(codes, counts, opts))
        s["llr"] = [_llr((g, c.N), case["ebn0"], c.K / c.N, seed * 64 + i)
                    for i, (c, g) in enumerate(zip(codes, counts))]
        run(s), run(s)  # the plan: tile sizes tuned, the iteration loop recorded
        return s
    if k == "ldpccc":
        J, L, p = case["J"], case["L"], case["p"]
        cc = pkg.LDPCCC(_shifts(J, L, p, 0, 3), p, case["I"], case["streams"], tanner=case["tanner"])
        for w, x in enumerate(_windows(case, cc.c, seed)[:-1]):
            cc.window(x, want_post=False)  # fills the pipeline: every later slot decides a frame
        return dict(case=case, cc=cc, llr=_windows(case, cc.c, seed, last=True))
    J, L, p = case["J"], case["L"], case["p"]
    zero = case.get("zero", 0)
    code = pkg.QCCode(_shifts(J, L, p, zero, 2), p)
    s = dict(case=case, code=code, seed=seed)
    if k == "decode":
        s["llr"] = _llr((case["gamma"], code.N), case["ebn0"], 1 - J / L, seed)
        if case["algo"] == "noms":
            s["params"] = _params(case["iters"], J * L, 5)
    elif k == "sim" and case["algo"] == "noms":
        s["params"] = _params(case["iters"], J * L, 5)
    elif k == "train":
        s["llr"] = _llr((case["frames"], code.N), case["ebn0"], 1 - J / L, seed)
        s["params"] = _params(case["T"], J * L, seed + 1)
    elif k == "encode":
        kk, _ = code.info_set()  # the encoder, built once for a code
        s["info"] = torch.randint(0, 2, (case["gamma"], kk), generator=_gen(seed), device="cuda", dtype=torch.uint8)
        code.encode(s["info"][:1])
    return s


class _Batch:
    """Owns a batch handle (and keeps its codes alive)."""

    def __init__(self, codes, counts, opts):
        self.codes, self.handle = codes, pkg.ldpc_batch_create(codes, counts, opts)

    def __del__(self):
        pkg.ldpc_batch_destroy(self.handle)


def _windows(case, c, seed, last=False):
    """Channel LLRs [streams][T][c]: enough windows to fill the pipeline, then one more."""
    lam = (2 if case["tanner"] else math.gcd(case["J"], case["L"]))
    n = (case["I"] * lam + case["T"] - 1) // case["T"] + 1
    shape = (case["streams"], case["T"], c)
    pick = [n - 1] if last else range(n)
    out = [_llr(shape, case["ebn0"], 1 - case["J"] / case["L"], seed * 1000 + w) for w in pick]
    return out[0] if last else out


# ---------------------------------------------------------------------------------------------- run
def run(s):
    case = s["case"]
    k = case["kind"]
    if k in ("decode", "sparse"):
        code, llr = s["code"], s["llr"]
        if case["algo"] == "noms":
            o = pkg.default_opts(max_iter=case["iters"], early_stop=int(case["early"]), algo=pkg.ALGO_NOMS,
                                 msg=MSG[case["msg"]], noms_params=s["params"].data_ptr())
            post = torch.empty_like(llr) if case["post"] else None
            hard = torch.empty(llr.shape, dtype=torch.uint8, device="cuda")
            it, ok = (torch.empty(llr.shape[0], dtype=torch.int32, device="cuda") for _ in range(2))
            pkg.ldpc_decode(code.handle, llr, o, post, hard, it, ok)
        else:
            post, hard, it, ok = code.decode(llr, max_iter=case["iters"], early_stop=case["early"],
                                             algo=ALGO[case["algo"]], msg=MSG[case["msg"]], want_post=case["post"])
        return {"post": post, "hard": hard, "iters": it, "ok": ok}
    if k == "sim":
        opt = dict(max_iter=case["iters"], early_stop=1, algo=ALGO[case["algo"]], msg=MSG[case["msg"]])
        if case["algo"] == "noms":
            opt["noms_params"] = s["params"].data_ptr()
        r = s["code"].ber_sim(case["ebn0"], seed=s["seed"], first_frame=0, max_frames=case["frames"],
                              target_frame_errors=1 << 60, gamma=case["gamma"], **opt)
        del r["seconds"]  # a wall-clock reading, not a result
        return r
    if k == "ldpccc":
        first, n, hard, post = s["cc"].window(s["llr"], want_post=case["post"])
        return {"n": n, "hard": hard, "post": post}
    if k == "batch":
        codes, counts = s["codes"], s["counts"]
        hard = [torch.empty((g, c.N), dtype=torch.uint8, device="cuda") for c, g in zip(codes, counts)]
        its, oks = ([torch.empty(g, dtype=torch.int32, device="cuda") for g in counts] for _ in range(2))
        pkg.ldpc_batch_decode(s["batch"].handle, s["llr"], hard, its, oks)
        return {"hard": hard, "iters": its, "ok": oks}
    if k == "train":
        loss, post = pkg.ldpc_noms_forward(s["code"].handle, s["llr"], s["params"], MSG[case["msg"]], case["ckpt"],
                                           CLIP, want_post=True)
        grad = torch.zeros_like(s["params"])
        pkg.ldpc_noms_backward(s["code"].handle, s["params"], grad)
        return {"loss": loss, "post": post, "grad": grad}
    cw = s["code"].encode(s["info"])
    return {"cw": cw, "llr": s["code"].channel_codewords(case["ebn0"], s["seed"], 0, cw)}


# --------------------------------------------------------------------------------------------- work
# operations per edge and iteration: sum-product evaluates the transform twice (about 24 operations
# each) and adds five times; the min-sum rules compare, select and add
OPS = {"sp": 53, "ms": 10, "noms": 14}


def work(case):
    k = case["kind"]
    if k == "batch":
        b = f = 0
        for J, L, p, g in _members(case):
            b += g * (L * p * 5 + 8)
            f += g * J * L * p * case["typ"] * OPS[case["algo"]]
        return {"bytes": b, "flops": f}
    if k == "sparse":
        N, E = case["N"], len(_random_rows(case["N"], case["M"], 1)[1])
        return {"bytes": case["gamma"] * (N * (5 + 4 * case["post"]) + 8) + 8 * E,
                "flops": case["gamma"] * E * case["typ"] * OPS[case["algo"]]}
    J, L, p = case["J"], case["L"], case["p"]
    N, E = L * p, J * L * p - case.get("zero", 0) * p
    if k == "decode":
        return {"bytes": case["gamma"] * (N * (5 + 4 * case["post"]) + 8),
                "flops": case["gamma"] * E * case["typ"] * OPS[case["algo"]]}
    if k == "sim":  # frames are drawn, decoded and counted on the device: only the counts leave
        return {"bytes": 48, "flops": case["frames"] * (E * case["typ"] * OPS[case["algo"]] + 60 * N)}
    if k == "ldpccc":
        c = N if case["tanner"] else N // math.gcd(J, L)
        g, T, I = case["streams"], case["T"], case["I"]
        return {"bytes": g * T * c * (5 + 4 * case["post"]), "flops": g * T * I * J * c * OPS["sp"]}
    if k == "train":
        return {"bytes": case["frames"] * N * 8 + 3 * case["T"] * J * L * 8,
                "flops": case["frames"] * case["T"] * E * 3 * OPS["noms"]}
    kk = N - J * p
    return {"bytes": case["gamma"] * (kk + 2 * N + 4 * N), "flops": case["gamma"] * (J * p * J * p / 16 + 60 * N)}


# -------------------------------------------------------------------------------------------- exact
def _phi(x):
    return torch.log1p(2.0 / torch.expm1(x))


class _Graph:
    """Edge tables of H: edges numbered row by row; rows padded with an absent edge E."""

    def __init__(self, rp, col, N):
        rp, col = np.asarray(rp, dtype=np.int64), np.asarray(col, dtype=np.int64)
        deg = np.diff(rp)
        M, E, dc = len(deg), len(col), int(deg.max())
        tab = np.full((M, dc), E, dtype=np.int64)
        pos = np.arange(E) - np.repeat(rp[:-1], deg)
        tab[np.repeat(np.arange(M), deg), pos] = np.arange(E)
        self.N, self.M, self.E, self.dc = N, M, E, dc
        self.tab = torch.from_numpy(tab).cuda()
        self.col = torch.from_numpy(col).cuda()


def _qc_rows(a, p):
    J, L = a.shape
    cols = []
    rp = [0]
    for j in range(J):
        ls = np.nonzero(a[j] >= 0)[0]
        c = ls[None, :] * p + (np.arange(p)[:, None] + a[j, ls][None, :]) % p
        cols.append(c.reshape(-1))
        rp += [rp[-1] + len(ls) * (r + 1) for r in range(p)]
    return np.asarray(rp), np.concatenate(cols)


def _check_sp(x):
    """alpha of rows whose messages are x [..., dc, F]; absent edges hold +inf (phi = 0, sign +)."""
    f = _phi(x.abs())
    sg = torch.where(x < 0, -1.0, 1.0)
    out = torch.empty_like(x)
    run_ = torch.zeros_like(x[..., 0, :])
    for l in range(x.shape[-2]):
        out[..., l, :] = run_
        run_ = run_ + f[..., l, :]
    run_ = torch.zeros_like(run_)
    for l in range(x.shape[-2] - 1, -1, -1):
        out[..., l, :] += run_
        run_ = run_ + f[..., l, :]
    return _phi(out).clamp(max=CLIP) * (sg.prod(dim=-2, keepdim=True) * sg)


def _min_other(x):
    """Minimum of |x| over the other edges of a row, and the sign of their product (sign(0) = +)."""
    a = x.abs()
    two, idx = torch.topk(a, 2, dim=-2, largest=False) if a.shape[-2] > 1 else (a.expand(*a.shape[:-2], 2, -1), None)
    m = two[..., 0:1, :].expand_as(a).clone()
    if idx is not None:
        m.scatter_(-2, idx[..., 0:1, :], two[..., 1:2, :])
    sg = torch.where(x < 0, -1.0, 1.0)
    return m, sg.prod(dim=-2, keepdim=True) * sg


def _bp(graph, mu, iters, early, algo, params=None, circ=None):
    """Algorithm 1 on frames mu [F][N] (64 bits): the posteriors [F][N]."""
    G = graph
    m = mu.t().contiguous()
    F = m.shape[1]
    big = float("inf")
    post = m.clone()
    beta = torch.cat([m[G.col], torch.full((1, F), big, dtype=m.dtype, device=m.device)])
    live = torch.ones(F, dtype=torch.bool, device=m.device)
    for it in range(iters):
        x = beta[G.tab]  # [M][dc][F]
        if algo == "sp":
            al = _check_sp(x)
        else:
            mag, sg = _min_other(x)
            if algo == "ms":
                al = mag.clamp(max=127.0) * sg
            else:
                wo = params[it][circ]  # [E][2]
                wo = torch.cat([wo, wo.new_zeros((1, 2))])[G.tab]
                al = (wo[..., 0:1] * mag - wo[..., 1:2]).clamp(min=0.0, max=CLIP) * sg
        alpha = torch.empty_like(beta)
        alpha[G.tab.reshape(-1)] = al.reshape(-1, F)
        alpha = alpha[:-1]
        tot = m.clone().index_add_(0, G.col, alpha)
        lim = 127.0 if algo == "ms" else CLIP
        beta[:-1] = (tot[G.col] - alpha).clamp(-lim, lim)
        new = tot if algo == "ms" else tot.clamp(-CLIP, CLIP)
        post = torch.where(live, new, post)
        if early:
            bad = torch.cat([(post < 0)[G.col], torch.zeros((1, F), dtype=torch.bool, device=m.device)])
            live = live & ((bad[G.tab].sum(dim=1) & 1) != 0).any(dim=0)
            if not live.any():
                break
    return post.t()


def _decode_exact(graph, case, llr, params=None, circ=None):
    algo = case["algo"]
    step = max(1, int(6e7 // graph.E))
    out = torch.empty(llr.shape, dtype=torch.float64, device=llr.device)
    for f in range(0, llr.shape[0], step):
        x = llr[f:f + step].double()
        x = (x * 4.0).round().clamp(-127, 127) if algo == "ms" else x.clamp(-CLIP, CLIP)
        y = _bp(graph, x, case["iters"], case["early"], algo, params, circ)
        out[f:f + step] = y * 0.25 if algo == "ms" else y
    return out


def _ldpccc_exact(case, seed):
    """Algorithm 2 on every stream (derived code, Sec. II-D): posteriors of the last window's decided frames."""
    J, L, p, I, S, T = (case[x] for x in ("J", "L", "p", "I", "streams", "T"))
    a = _shifts(J, L, p, 0, 3)
    lam = math.gcd(J, L)
    Jb, Lb, ms = J // lam, L // lam, lam - 1
    c = Lb * p
    frames = torch.cat(_windows(case, c, seed), dim=1)
    mu, alpha, beta = {}, {}, {}
    r = np.arange(p)
    at = {(j, l): torch.from_numpy((l % Lb) * p + (r + a[j, l]) % p).cuda() for j in range(J) for l in range(L)}
    post = []
    total = frames.shape[1]
    for t in range(total):
        mu[t] = frames[:, t].double().clamp(-CLIP, CLIP).t().contiguous()
        alpha[t] = mu[t].new_zeros((J, c, S))
        beta[t] = mu[t].expand(J, c, S).clone()
        for i in range(I):
            R = t - i * lam
            if R < 0:
                break
            ty = R % lam
            for j in range(ty * Jb, (ty + 1) * Jb):
                x = mu[t].new_full((p, L, S), float("inf"))
                fr = [R - (ty - l // Lb) % lam for l in range(L)]
                for l in range(L):
                    if fr[l] >= 0:
                        x[:, l] = beta[fr[l]][j, at[j, l]]
                al = _check_sp(x)
                for l in range(L):
                    if fr[l] >= 0:
                        alpha[fr[l]][j, at[j, l]] = al[:, l]
        for i in range(I):
            f = t - i * lam - ms
            if f < 0:
                break
            tot = mu[f] + alpha[f].sum(dim=0)
            beta[f] = (tot - alpha[f]).clamp(-CLIP, CLIP)
            if i == I - 1:
                if t >= total - T:
                    post.append(tot.clamp(-CLIP, CLIP).t())
                del mu[f], alpha[f], beta[f]
    return torch.stack(post, dim=1)


def _train_exact(case, seed):
    """Loss, last posteriors and parameter gradient of the unrolled learned min-sum, in 64 bits by autograd."""
    J, L, p, T, B = (case[x] for x in ("J", "L", "p", "T", "frames"))
    N = L * p
    a = _shifts(J, L, p, 0, 2)
    G = _Graph(*_qc_rows(a, p), N)
    circ = torch.arange(J, device="cuda").repeat_interleave(p * L) * L + G.col // p
    par = _params(T, J * L, seed + 1).double().requires_grad_(True)
    llr = _llr((B, N), case["ebn0"], 1 - J / L, seed)
    loss = 0.0
    posts = []
    step = max(1, int(8e6 // G.E))
    for f in range(0, B, step):
        m = llr[f:f + step].double().clamp(-CLIP, CLIP).t().contiguous()
        beta = m[G.col]
        part = 0.0
        for it in range(T):
            x = beta[G.tab]
            two, idx = torch.topk(x.abs(), 2, dim=1, largest=False)
            first = torch.zeros_like(x, dtype=torch.bool).scatter_(1, idx[:, :1], True)
            mag = torch.where(first, two[:, 1:2], two[:, 0:1])
            sg = torch.where(x < 0, -1.0, 1.0)
            sg = sg.prod(dim=1, keepdim=True) * sg
            wo = par[it][circ][G.tab]
            al = ((wo[..., 0:1] * mag - wo[..., 1:2]).clamp(min=0.0, max=CLIP) * sg.detach()).reshape(G.E, -1)
            tot = m.index_add(0, G.col, al)
            beta = (tot[G.col] - al).clamp(-CLIP, CLIP)
            part = part + torch.nn.functional.softplus(-tot).sum()
        part = part / (T * N * B)
        part.backward()
        loss += float(part.detach())
        posts.append(tot.detach().t())
    return {"loss": torch.tensor([loss], dtype=torch.float64), "post": torch.cat(posts), "grad": par.grad}


def _channel_exact(case, seed, cw):
    """mu = 2 (x + sigma g) / sigma^2, g Box-Muller normals of Philox4x32-10 words (the library's counters)."""
    B, N = cw.shape
    Q = (N + 3) // 4
    M32 = 0xFFFFFFFF
    q = torch.arange(Q, dtype=torch.int64, device="cuda")[None, :].expand(B, Q)
    f = torch.arange(B, dtype=torch.int64, device="cuda")[:, None].expand(B, Q)

    def mul(k, x):  # the high and low words of k * x without leaving 63 bits
        lo, hi = (x & 0xFFFF) * k, (x >> 16) * k
        s = (lo >> 16) + (hi & M32)
        return ((hi >> 32) << 16) + (s >> 16) & M32, ((s & 0xFFFF) << 16 | lo & 0xFFFF) & M32

    c = [q, f, torch.zeros_like(q), torch.zeros_like(q)]
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    u = [((w >> 9).double() + 0.5) * 2.0 ** -23 for w in c]
    g = torch.empty((B, Q, 4), dtype=torch.float64, device="cuda")
    for e in (0, 2):
        rho = torch.sqrt(-2.0 * torch.log(u[e]))
        g[..., e] = rho * torch.cos(2 * math.pi * u[e + 1])
        g[..., e + 1] = rho * torch.sin(2 * math.pi * u[e + 1])
    sigma = math.sqrt(1.0 / (2.0 * (1 - case["J"] / case["L"]) * 10.0 ** (case["ebn0"] / 10.0)))
    return 2.0 / sigma ** 2 * ((1.0 - 2.0 * cw.double()) + sigma * g.reshape(B, Q * 4)[:, :N])


def _encode_exact(case, seed):
    """The codewords of the drawn information bits: parity positions by elimination over GF(2), right to left."""
    J, L, p = case["J"], case["L"], case["p"]
    N, M = L * p, J * p
    rp, col = _qc_rows(_shifts(J, L, p, 0, 2), p)
    H = torch.zeros((M, N), dtype=torch.bool, device="cuda")
    H[torch.arange(M, device="cuda").repeat_interleave(L), torch.from_numpy(col).cuda()] = True
    A = H.flip(1).clone()
    piv, row = [], 0
    for n in range(N):
        if row == M:
            break
        hit = torch.nonzero(A[row:, n])
        if not len(hit):
            continue
        r = row + int(hit[0])
        if r != row:
            A[[row, r]] = A[[r, row]]
        other = A[:, n].clone()
        other[row] = False
        A[other] ^= A[row]
        piv.append(N - 1 - n)
        row += 1
    A = A[:row].flip(1)
    par = torch.tensor(piv, device="cuda")
    info = torch.ones(N, dtype=torch.bool, device="cuda")
    info[par] = False
    u = torch.randint(0, 2, (case["gamma"], int(info.sum())), generator=_gen(seed), device="cuda", dtype=torch.uint8)
    cw = torch.zeros((case["gamma"], N), dtype=torch.uint8, device="cuda")
    cw[:, info] = u
    cw[:, par] = ((u.float() @ A[:, info].float().t()) % 2).to(torch.uint8)
    return cw


def exact(case, seed):
    k = case["kind"]
    if k in ("decode", "sparse"):
        if not case["post"]:
            return None
        par = circ = None
        if k == "sparse":
            rp, col = _random_rows(case["N"], case["M"], 1)
            N, rate = case["N"], 1 - case["M"] / case["N"]
        else:
            a = _shifts(case["J"], case["L"], case["p"], case["zero"], 2)
            rp, col = _qc_rows(a, case["p"])
            N, rate = case["L"] * case["p"], 1 - case["J"] / case["L"]
        G = _Graph(rp, col, N)
        if case["algo"] == "noms":
            J, L, p = case["J"], case["L"], case["p"]
            deg = torch.from_numpy(np.diff(rp)).cuda()
            circ = (torch.arange(J * p, device="cuda") // p).repeat_interleave(deg) * L + G.col // p
            par = _params(case["iters"], J * L, 5).double()
        return {"post": _decode_exact(G, case, _llr((case["gamma"], N), case["ebn0"], rate, seed), par, circ),
                "hard": None, "iters": None, "ok": None}
    if k == "ldpccc":
        if case["tanner"] or not case["post"] or case["I"] * case["J"] * case["L"] * case["T"] > 1 << 18:
            return None
        return {"n": None, "hard": None, "post": _ldpccc_exact(case, seed)}
    if k == "train":
        return _train_exact(case, seed)
    if k == "encode":
        if case["J"] * case["p"] > 3072:
            return None
        cw = _encode_exact(case, seed)
        return {"cw": cw, "llr": _channel_exact(case, seed, cw)}
    return None  # a simulation's counts and a mixed batch's decisions are whole numbers
