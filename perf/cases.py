"""What the detectors are timed on: the calls a receiver or a simulation makes.

Every case is one call of a public entry point of
paper_2002_09561_gb300.mdx on inputs drawn on the GPU with the system model
y = H s + n (H i.i.d. CN(0, 1), uniform QAM symbols, noise of variance
10^(-SNR/10) per complex receive entry), the same distributions as
paper_2002_09561_gb300.workload.  Sizes are those of the benchmark's
workloads and of the tests.  Receivers that only need decisions ask for no
search statistics; the fixed-complexity K-best runs with them, as a
simulation does.
"""

import math

import numpy as np
import torch

from paper_2002_09561_gb300 import mdx, train

ANTENNAS, QAMS = (8, 16, 32, 64, 100), (4, 16, 64)


def listed():
    return [
        # a real-time receiver with one subcarrier in hand: launches and latency
        dict(name="sd-one-16x16", kind="sd", n_rx=16, n_tx=16, qam=16, snr_lo=18.0, snr_hi=18.0, batch=1),
        # the default benchmark: exact detection from the network's radius and first leaf, 4..20 dB
        dict(name="sd-learned-16x16", kind="sd_learned", n_rx=16, n_tx=16, qam=16, snr_lo=4.0, snr_hi=20.0,
             batch=100_000),
        # exact detection with the paper's radius, more receive than transmit antennas, a ragged batch
        dict(name="sd-12x9-64qam", kind="sd", n_rx=12, n_tx=9, qam=64, snr_lo=20.0, snr_hi=28.0, batch=10_007),
        # exact detection above 32 real rows
        dict(name="sd-24x24", kind="sd", n_rx=24, n_tx=24, qam=16, snr_lo=18.0, snr_hi=18.0, batch=8_000),
        # fixed-complexity detection over the benchmark's sweep
        dict(name="kbest64-16x16", kind="kbest", n_rx=16, n_tx=16, qam=16, snr_lo=4.0, snr_hi=20.0, K=64,
             batch=100_000),
        # the paper's 16x16 64-QAM K-best on the complex tree (481 visited nodes)
        dict(name="kbest32-complex-16x16", kind="kbest_complex", n_rx=16, n_tx=16, qam=64, snr_lo=16.0, snr_hi=28.0,
             K=32, batch=20_000),
        # massive MIMO: the hybrid detector with the network's radius
        dict(name="hybrid32-100x100", kind="hybrid_learned", n_rx=100, n_tx=100, qam=64, snr_lo=20.0, snr_hi=32.0,
             K=32, depth=4, batch=4_000),
        # a base station's uneven mix: antennas, modulations and detectors differ by request
        dict(name="mixed-10k", kind="mixed", snr_lo=6.0, snr_hi=30.0, K=64, budget=20_000, batch=10_000),
        # the QR preprocessing alone, as another detector's front end calls it
        dict(name="qr-64x64", kind="qr", n_rx=64, n_tx=64, batch=3_000),
        # the linear control: MMSE
        dict(name="mmse-16x16", kind="mmse", n_rx=16, n_tx=16, qam=16, snr_lo=4.0, snr_hi=20.0, batch=100_000),
        # detection of vectors that arrive in pinned host memory
        dict(name="host-kbest16-8x8", kind="kbest_host", n_rx=8, n_tx=8, qam=64, snr_lo=16.0, snr_hi=28.0, K=16,
             batch=50_000),
        # one training step of the radius network (features, forward, backward, Adam)
        dict(name="train-16x16", kind="train", n_rx=16, n_tx=16, qam=16, snr_lo=8.0, snr_hi=20.0, batch=4_096),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sd", "sd", "sd_learned", "sd_large", "kbest", "kbest", "kbest_complex", "hybrid",
                       "hybrid_learned", "mixed", "qr", "qr", "zf", "mmse", "kbest_host", "train"])
    qam = rng.choice(QAMS)
    if kind == "sd":
        n = rng.randint(2, 16)
        lo = {4: 10.0, 16: 17.0, 64: 23.0}[qam] + rng.uniform(0.0, 6.0)
        return dict(kind="sd", n_rx=n + rng.randint(0, 4), n_tx=n, qam=qam, snr_lo=lo, snr_hi=lo + rng.uniform(0.0, 6.0),
                    batch=_log_int(rng, 1, 30_000))
    if kind == "sd_learned":
        return dict(kind=kind, n_rx=16, n_tx=16, qam=16, snr_lo=rng.uniform(4.0, 14.0), snr_hi=20.0,
                    batch=_log_int(rng, 1_000, 90_000))
    if kind == "sd_large":
        n = rng.randint(17, 24)
        lo = rng.uniform(18.0, 22.0)
        return dict(kind="sd", n_rx=n + rng.randint(0, 4), n_tx=n, qam=16, snr_lo=lo, snr_hi=lo + rng.uniform(0.0, 4.0),
                    batch=_log_int(rng, 100, 7_000))
    if kind in ("kbest", "kbest_host"):
        n, K = rng.randint(2, 32 if kind == "kbest" else 16), _log_int(rng, 4, 200 if kind == "kbest" else 32)
        most = max(2, min(60_000, int(6e8 / (2 * n * K * math.isqrt(qam) * (1 + n / 8)))))
        return dict(kind=kind, n_rx=n + rng.randint(0, 4), n_tx=n, qam=qam, snr_lo=8.0 + 4.0 * math.log2(qam) - 8.0,
                    snr_hi=8.0 + 4.0 * math.log2(qam), K=K, batch=_log_int(rng, 1, most))
    if kind == "kbest_complex":
        n, K = rng.randint(2, 16), _log_int(rng, 4, 48)
        return dict(kind=kind, n_rx=n + rng.randint(0, 4), n_tx=n, qam=qam, snr_lo=16.0, snr_hi=28.0, K=K,
                    batch=_log_int(rng, 1, max(2, min(20_000, int(6e8 / (n * K * qam))))))
    if kind == "hybrid":
        n = rng.randint(8, 96)
        return dict(kind=kind, n_rx=min(n + rng.randint(0, 8), 100), n_tx=n, qam=rng.choice((16, 64)), snr_lo=22.0,
                    snr_hi=32.0, K=_log_int(rng, 8, 48), depth=rng.randint(2, 4), batch=_log_int(rng, 100, 2_000))
    if kind == "hybrid_learned":
        return dict(kind=kind, n_rx=100, n_tx=100, qam=64, snr_lo=rng.uniform(20.0, 26.0), snr_hi=32.0,
                    K=_log_int(rng, 8, 32), depth=4, batch=_log_int(rng, 100, 3_500))
    if kind == "mixed":
        return dict(kind=kind, snr_lo=rng.uniform(6.0, 12.0), snr_hi=30.0, K=_log_int(rng, 16, 64), budget=20_000,
                    batch=_log_int(rng, 200, 9_000))
    if kind == "qr":
        n = rng.randint(2, 100)
        return dict(kind=kind, n_rx=n + rng.randint(0, 8), n_tx=n,
                    batch=_log_int(rng, 1, max(2, min(60_000, int(2e9 / n ** 3)))))
    if kind in ("zf", "mmse"):
        n = rng.randint(2, 32)
        return dict(kind=kind, n_rx=n + rng.randint(0, 4), n_tx=n, qam=qam, snr_lo=8.0, snr_hi=24.0,
                    batch=_log_int(rng, 1, min(90_000, int(3e8 / n ** 3))))
    return dict(kind="train", n_rx=16, n_tx=16, qam=16, snr_lo=rng.uniform(8.0, 12.0), snr_hi=20.0,
                batch=_log_int(rng, 256, 8_000))


# ----------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _points(q, qam):
    """Complex unit-energy points of the indices q = k_re P + k_im."""
    p = math.isqrt(qam)
    a = math.sqrt(3.0 / (2.0 * (qam - 1)))
    return torch.complex(((2 * (q // p) - (p - 1)) * a).double(), ((2 * (q % p) - (p - 1)) * a).double())


def _noise_var(case, count):
    """The SNR points snr_lo .. snr_hi in nine equal steps, interleaved."""
    snr = case["snr_lo"] + (case["snr_hi"] - case["snr_lo"]) / 8.0 * (torch.arange(count, device="cuda") % 9).double()
    return torch.pow(10.0, -snr / 10.0)


def _channels(g, count, n_rx, n_tx):
    return torch.randn((count, n_rx, n_tx, 2), generator=g, device="cuda", dtype=torch.float64) * math.sqrt(0.5)


def _observe(g, H, q, qam, nv):
    """y = H s + n of channels H [B][N][M][2] and symbol indices q [B][M]."""
    s = _points(q, qam)
    y = torch.view_as_real(torch.einsum("bnm,bm->bn", torch.view_as_complex(H), s))
    w = torch.randn(y.shape, generator=g, device="cuda", dtype=torch.float64)
    return (y + w * torch.sqrt(nv / 2.0)[:, None, None]).contiguous()


def _inputs(case, seed):
    g, B = _gen(seed), case["batch"]
    H = _channels(g, B, case["n_rx"], case["n_tx"])
    q = torch.randint(0, case["qam"], (B, case["n_tx"]), generator=g, device="cuda")
    nv = _noise_var(case, B)
    return H, _observe(g, H, q, case["qam"], nv), nv, q


def _mixed_table(case, seed):
    """The requests: every (antennas, modulation, detector) class equally often, in a random order."""
    B = case["batch"]
    i = np.random.RandomState(int(seed) % (1 << 31)).permutation(B)
    n = np.asarray(ANTENNAS)[i % 5]
    qam = np.asarray(QAMS)[i // 5 % 3]
    return mdx.make_requests(n, n, qam, i // 15 % 2, K=case["K"], budget=case["budget"])


def _mixed_inputs(case, seed):
    g, B = _gen(seed), case["batch"]
    reqs = _mixed_table(case, seed)
    nv = _noise_var(case, B)
    nv = nv[torch.randperm(B, generator=g, device="cuda")].contiguous()
    last = reqs[-1]
    H = torch.randn(int(last["h_offset"] + 2 * last["n_rx"] * last["n_tx"]), generator=g, device="cuda",
                    dtype=torch.float64) * math.sqrt(0.5)
    y = torch.empty(int(last["y_offset"] + 2 * last["n_rx"]), device="cuda", dtype=torch.float64)
    for n in ANTENNAS:
        for qam in QAMS:
            at = np.flatnonzero((reqs["n_tx"] == n) & (reqs["qam"] == qam))
            if not at.size:
                continue
            ho = torch.from_numpy(reqs["h_offset"][at].copy()).cuda()[:, None] + torch.arange(2 * n * n, device="cuda")
            yo = torch.from_numpy(reqs["y_offset"][at].copy()).cuda()[:, None] + torch.arange(2 * n, device="cuda")
            q = torch.randint(0, qam, (at.size, n), generator=g, device="cuda")
            Hc = H[ho].view(at.size, n, n, 2)
            y[yo] = _observe(g, Hc, q, qam, nv[torch.from_numpy(at).cuda()]).view(at.size, -1)
    return reqs, H, y, nv


def prepare(case, seed):
    kind, B = case["kind"], case["batch"]
    if kind == "mixed":
        reqs, H, y, nv = _mixed_inputs(case, seed)
        ctx = mdx.Context(0, B, max(ANTENNAS), max(ANTENNAS))
        nsym = int((reqs["sym_offset"] + reqs["n_tx"]).max())
        out = (torch.empty(nsym, dtype=torch.uint8, device="cuda"), torch.empty(B, dtype=torch.float64, device="cuda"),
               torch.empty(B, dtype=torch.int32, device="cuda"), None)
        return dict(kind=kind, ctx=ctx, reqs=reqs, H=H, y=y, nv=nv, out=out)
    if kind == "qr":
        g = _gen(seed)
        H = _channels(g, B, case["n_rx"], case["n_tx"])
        y = torch.randn((B, case["n_rx"], 2), generator=g, device="cuda", dtype=torch.float64)
        return dict(kind=kind, ctx=mdx.Context(0, B, case["n_rx"], case["n_tx"]), H=H, y=y)
    H, y, nv, q = _inputs(case, seed)
    n_rx, n_tx, qam = case["n_rx"], case["n_tx"], case["qam"]
    ctx = mdx.Context(0, B, n_rx, n_tx)
    st = dict(kind=kind, ctx=ctx, H=H, y=y, nv=nv)
    if kind == "train":
        train.load_model(ctx, n_tx, qam, max_train_batch=B)
        # the traces: the transmitted point stands for the exact detector's answer
        r = torch.view_as_complex(y) - torch.einsum("bnm,bm->bn", torch.view_as_complex(H), _points(q, qam))
        st.update(params=mdx.make_params(n_rx, n_tx, qam), sym=q.to(torch.uint8),
                  metric=(r.real ** 2 + r.imag ** 2).sum(1).contiguous())
        return st
    flags, radius, algo, stats = 0, math.inf, "kbest", None
    if kind.endswith("_learned"):
        train.load_model(ctx, n_tx, qam)
        flags |= mdx.MDX_LEARNED_RADIUS | (mdx.MDX_LEARNED_ORDER if kind == "sd_learned" else 0)
    if kind.startswith(("sd", "hybrid")):
        radius, algo = "paper", "sd" if kind.startswith("sd") else "hybrid"
    elif kind in ("zf", "mmse"):
        flags, algo = mdx.MDX_LINEAR_MMSE if kind == "mmse" else 0, "linear"
    else:
        flags = mdx.MDX_COMPLEX_TREE if kind == "kbest_complex" else 0
    st.update(algo=algo, params=mdx.make_params(n_rx, n_tx, qam, radius=radius, K=case.get("K", 16),
                                                depth=case.get("depth", 4), flags=flags))
    if kind == "kbest_host":
        pin = [t.cpu().pin_memory() for t in (H, y, nv)]
        outs = [torch.empty(s, dtype=t, pin_memory=True) for s, t in
                (((B, n_tx), torch.uint8), ((B,), torch.float64), ((B,), torch.int32))]
        return dict(kind=kind, algo=algo, ctx=ctx, params=st["params"], keep=pin + outs,
                    host=[t.numpy() for t in pin], out=[t.numpy() for t in outs])
    if algo == "kbest":
        stats = torch.empty((B, mdx.STATS), dtype=torch.int64, device="cuda")
    st["out"] = (torch.empty((B, n_tx), dtype=torch.uint8, device="cuda"),
                 torch.empty(B, dtype=torch.float64, device="cuda"), torch.empty(B, dtype=torch.int32, device="cuda"),
                 stats)
    return st


def run(st):
    """One call; its outputs (detectors: symbols, metrics, per-vector status and, for K-best, statistics)."""
    kind = st["kind"]
    if kind == "qr":
        return mdx.qr(st["ctx"], st["H"], st["y"])
    if kind == "train":
        return mdx.mlp_train_step(st["ctx"], st["params"], st["H"], st["y"], st["nv"], st["sym"], st["metric"],
                                  lr=1e-3, update=True, want_grad=True)
    if kind == "mixed":
        return mdx.detect_mixed(st["ctx"], st["reqs"], st["H"], st["y"], st["nv"], out=st["out"])
    if kind == "kbest_host":
        mdx.detect_host(st["algo"], st["ctx"], st["params"], *st["host"], *st["out"])
        return st["out"]
    return mdx.detect(st["algo"], st["ctx"], st["params"], st["H"], st["y"], st["nv"], out=st["out"])


# ----------------------------------------------------------------- work


def _qr_flops(n_rx, n_tx):
    return 8.0 * (n_rx * n_tx ** 2 - n_tx ** 3 / 3.0)


def _kbest_flops(n_tx, qam, K, cplx=False):
    """Surviving nodes times 2 (n - 1 - i) + 4 P per real row (both rows of a complex level)."""
    n, p, nodes, total = 2 * n_tx, math.isqrt(qam), 1, 0.0
    for i in range(n - 1, -1, -1):
        total += min(nodes, K) * (2 * (n - 1 - i) + 4 * p)
        if not cplx or i % 2 == 0:
            nodes = min(min(nodes, K) * (qam if cplx else p), 1 << 30)
    return total


def work(case):
    """Bytes: every input read once, every output written once.  Flops: the QR in complex Householder
    form, the search's own count (SD and hybrid: one descent, which no search can do without)."""
    kind, B = case["kind"], case["batch"]
    if kind == "mixed":
        i = np.arange(B)
        n, qam, kb = np.asarray(ANTENNAS)[i % 5], np.asarray(QAMS)[i // 5 % 3], i // 15 % 2
        flops = sum(_qr_flops(int(a), int(a)) + _kbest_flops(int(a), int(q), case["K"] if k else 1)
                    for a, q, k in zip(n, qam, kb))
        return {"bytes": float((16 * n * n + 16 * n + n + 8 + 8 + 4).sum()), "flops": float(flops)}
    n_rx, n_tx = case["n_rx"], case["n_tx"]
    io = 16.0 * n_rx * n_tx + 16.0 * n_rx
    if kind == "qr":
        return {"bytes": B * (io + 8.0 * (4 * n_tx * n_tx + 2 * n_tx)), "flops": B * _qr_flops(n_rx, n_tx)}
    if kind == "train":
        d_in, d_out = mdx.mlp_dims(n_tx, case["qam"])
        weights = mdx.mlp_param_count(n_tx, case["qam"])
        gemm = 2.0 * (d_in * 256 + 256 * 256 + 256 * d_out)
        # gradient written; weights and both moments read and written
        return {"bytes": B * (io + 8 + n_tx + 8) + 28.0 * weights + 8,
                "flops": B * (_qr_flops(n_rx, n_tx) + 3.0 * gemm)}
    io += 8.0 + n_tx + 8 + 4
    n = 2 * n_tx
    if kind in ("kbest", "kbest_complex"):
        io += 40.0
    if kind in ("zf", "mmse"):
        search = 2.0 * n * n + (n ** 3 / 3.0 + n ** 3 if kind == "mmse" else 0.0)
    else:
        search = _kbest_flops(n_tx, case["qam"], case["K"] if kind.startswith("kbest") else 1, kind == "kbest_complex")
    if kind == "sd_learned" or kind == "hybrid_learned":
        d_in, d_out = mdx.mlp_dims(n_tx, case["qam"])
        search += 2.0 * (d_in * 256 + 256 * 256 + 256 * d_out)
    return {"bytes": B * io, "flops": B * (_qr_flops(n_rx, n_tx) + search)}


# ----------------------------------------------------------------- exact answers, plain torch in 64 bits


def _qr64(H, y):
    """Real interleaved R [B][n][n] and ybar [B][n] by complex Householder reflections in torch."""
    A = torch.cat([torch.view_as_complex(H), torch.view_as_complex(y)[..., None]], 2)
    M = H.shape[2]
    for k in range(M):
        x = A[:, k:, k].clone()
        norm = torch.linalg.vector_norm(x, dim=1)
        x0 = x[:, 0].clone()
        ph = torch.where(x0.abs() > 0, x0 / x0.abs().clamp_min(1e-300), torch.ones_like(x0))
        x[:, 0] += ph * norm
        vv = (x.real ** 2 + x.imag ** 2).sum(1).clamp_min(1e-300)
        w = torch.einsum("br,brc->bc", x.conj(), A[:, k:, k:]) * (2.0 / vv)[:, None]
        A[:, k:, k:] -= x[:, :, None] * w[:, None, :]
        A[:, k, k:] *= (-ph.conj())[:, None]
    A = torch.cat([torch.triu(A[:, :M, :M]), A[:, :M, M:]], 2)
    n = 2 * M
    R = torch.zeros((A.shape[0], n, n), dtype=torch.float64, device=A.device)
    R[:, 0::2, 0::2] = R[:, 1::2, 1::2] = A[..., :M].real
    R[:, 0::2, 1::2], R[:, 1::2, 0::2] = -A[..., :M].imag, A[..., :M].imag
    return R.triu_(), torch.view_as_real(A[:, :, M].contiguous()).reshape(-1, n).contiguous()


def _levels(qam):
    p = math.isqrt(qam)
    return (2.0 * torch.arange(p, device="cuda", dtype=torch.float64) - (p - 1)) * math.sqrt(3.0 / (2.0 * (qam - 1)))


def _kbest64(R, yb, qam, K, cplx):
    """Metric of the best leaf of K-best, ties to the lower parent rank, then the lower child."""
    B, n = yb.shape
    lev = _levels(qam)
    p = lev.numel()
    path = torch.zeros((B, 1, 0), dtype=torch.float64, device="cuda")  # levels of rows i+1 .. n-1
    ped = torch.zeros((B, 1), dtype=torch.float64, device="cuda")
    for i in range(n - 1, -1, -1):
        c = yb[:, i, None] - torch.einsum("bsj,bj->bs", path, R[:, i, i + 1:])
        cost = ped[..., None] + (c[..., None] - R[:, i, i, None, None] * lev) ** 2  # [B][S][p]
        S = ped.shape[1]
        if cplx and i % 2:  # the level's imaginary row: keep every child until its real row is fixed
            path = torch.cat([lev.expand(B, S, p)[..., None], path[:, :, None, :].expand(B, S, p, path.shape[2])], 3)
            path, ped = path.reshape(B, S * p, -1), cost.reshape(B, S * p)
            continue
        if cplx:  # children of a node in the order q = k_re P + k_im
            cost = cost.view(B, S // p, p, p).transpose(2, 3).reshape(B, -1)
            at = torch.arange(S * p, device="cuda").view(S // p, p, p).transpose(1, 2).reshape(-1)
        else:
            cost, at = cost.reshape(B, -1), torch.arange(S * p, device="cuda")
        ped, order = torch.sort(cost, dim=1, stable=True)
        ped, order = ped[:, :K].contiguous(), at[order[:, :K]]
        up = torch.gather(path, 1, (order // p)[..., None].expand(-1, -1, path.shape[2]))
        path = torch.cat([lev[order % p][..., None], up], 2)
    return ped[:, 0]


def _linear64(R, yb, nv, qam, mmse):
    if mmse:
        G = R.mT @ R + nv[:, None, None] * torch.eye(R.shape[1], device="cuda", dtype=torch.float64)
        x = torch.cholesky_solve(R.mT @ yb[..., None], torch.linalg.cholesky(G))[..., 0]
    else:
        x = torch.linalg.solve_triangular(R, yb[..., None], upper=True)[..., 0]
    lev = _levels(qam)
    k = torch.round((x / lev[-1] + 1.0) * (0.5 * (lev.numel() - 1))).clamp(0, lev.numel() - 1).long()
    r = yb - torch.einsum("bij,bj->bi", R, lev[k])
    return (r * r).sum(1)


def _ml64(H, y, qam):
    """Smallest ||y - H s||^2 over every s (few antennas only), less the part of y outside H's columns."""
    B, N, M = H.shape[0], H.shape[1], H.shape[2]
    R, yb = _qr64(H, y)
    code = torch.arange(qam ** M, device="cuda")
    q = torch.stack([code // qam ** m % qam for m in range(M)], 1)
    s = torch.view_as_real(_points(q, qam)).reshape(-1, 2 * M)
    best = torch.empty(B, dtype=torch.float64, device="cuda")
    step = max(1, int(2e8) // (s.shape[0] * 2 * M))
    for b in range(0, B, step):
        r = yb[b:b + step, None, :] - torch.einsum("bij,sj->bsi", R[b:b + step], s)
        best[b:b + step] = (r * r).sum(2).min(1).values
    return best


def _train64(case, H, y, nv, q, params):
    """Pinball and cross-entropy losses and the gradient of the two-hidden-layer network, by autograd."""
    n_tx, qam = case["n_tx"], case["qam"]
    n, p = 2 * n_tx, math.isqrt(qam)
    d_in, d_out = mdx.mlp_dims(n_tx, qam)
    R, yb = _qr64(H, y)
    x = torch.zeros((H.shape[0], d_in), dtype=torch.float64, device="cuda")
    at = 0
    for c in range(n):
        x[:, at:at + c + 1] = R[:, :c + 1, c]
        at += c + 1
    x[:, at:at + n] = yb
    x[:, at + n] = -10.0 * torch.log10(nv) / 30.0
    w = params.double().cuda().requires_grad_(True)
    sizes = [256 * d_in, 256, 256 * 256, 256, d_out * 256, d_out]
    w1, b1, w2, b2, w3, b3 = torch.split(w, sizes)
    h = torch.relu(x @ w1.view(256, d_in).T + b1)
    h = torch.relu(h @ w2.view(256, 256).T + b2)
    o = h @ w3.view(d_out, 256).T + b3
    r = torch.view_as_complex(y) - torch.einsum("bnm,bm->bn", torch.view_as_complex(H), _points(q, qam))
    e = torch.log((r.real ** 2 + r.imag ** 2).sum(1) / nv) - o[:, 0]
    pin = torch.where(e >= 0, 0.9 * e, -0.1 * e).mean()
    k = torch.stack([q // p, q % p], 2).reshape(-1)
    ce = torch.nn.functional.cross_entropy(o[:, 1:1 + n * p].reshape(-1, p), k)
    (pin + 0.2 * ce).backward()
    return torch.stack([pin, ce]).detach(), w.grad


def exact(case, seed):
    """What run() returns for these inputs in 64 bits.  Searches whose answer plain torch cannot find in
    seconds (exact detection of many antennas, the hybrid, the uneven mix) have none."""
    kind, B = case["kind"], case["batch"]
    if kind == "qr":
        g = _gen(seed)
        H = _channels(g, B, case["n_rx"], case["n_tx"])
        y = torch.randn((B, case["n_rx"], 2), generator=g, device="cuda", dtype=torch.float64)
        return list(_qr64(H, y))
    if kind == "mixed" or kind.startswith("hybrid"):
        return None
    qam, M = case["qam"], case["n_tx"]
    if kind.startswith("sd") and B * float(qam) ** M * M > 2e9:
        return None
    H, y, nv, q = _inputs(case, seed)
    if kind == "train":
        params = torch.from_numpy(np.load(train.model_path(M, qam)))
        return list(_train64(case, H, y, nv, q, params))
    if kind.startswith("sd"):
        return [None, _ml64(H, y, qam), None]
    cplx = kind == "kbest_complex"
    step = B if not kind.startswith("kbest") else max(1, int(2e8) // (case["K"] * (qam if cplx else math.isqrt(qam)) * M))
    parts = []
    for b in range(0, B, step):
        R, yb = _qr64(H[b:b + step], y[b:b + step])
        if kind in ("zf", "mmse"):
            parts.append(_linear64(R, yb, nv[b:b + step], qam, kind == "mmse"))
        else:
            parts.append(_kbest64(R, yb, qam, case["K"], cplx))
    metric = torch.cat(parts)
    if kind == "kbest_host":
        return [None, metric.cpu().numpy(), None]
    return [None, metric, None] + ([None] if kind.startswith("kbest") else [])
