"""The work that a user of this library has it do, as cases that can be timed: searches from one
query to a full batch, in the encodings and options of the benchmark's workloads, the encoding of a
database, the graph builds, and the learning of the projections.

Inputs are drawn on the GPU from the Gaussian mixtures that workloads.py describes (database and
queries share a decaying spectrum; out-of-distribution queries are shifted and rotated).  What a
search case holds before the call (projection, stores, graph) is made from plain torch arithmetic and
the library's bit-reproducible parts (LVQ encoding around a given mean, graph build), so that the same
seed always gives the same index.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2312_16335_gb300 as lv

COMPONENTS = 1000
PREC = {"fp32": lv.PREC_FP32, "bf16": lv.PREC_BF16, "fp8": lv.PREC_FP8, "tf32x3": lv.PREC_TF32X3}


def listed():
    return [
        # One query against a small index (10k x 128, k = 10, L = 50, rerank 50: the repository's
        # parity workload): an interactive lookup, where the launches and one walk's latency count.
        {"name": "search_one_10k_128", "kind": "search", "n": 10000, "D": 128, "d": 32, "bits": 8, "R": 32,
         "L_build": 64, "metric": "ip", "graph": "primary", "m": 1, "k": 10, "L": 50, "rerank": 50, "hops": 0,
         "width": 1, "projection": "fp32", "uneven": False, "host": False},
        # A server's micro-batch: 100 queries that arrived together, on a 200k index.
        {"name": "search_online_200k_768", "kind": "search", "n": 200000, "D": 768, "d": 160, "bits": 8, "R": 64,
         "L_build": 128, "metric": "ip", "graph": "primary", "m": 100, "k": 10, "L": 128, "rerank": 128, "hops": 0,
         "width": 2, "projection": "bf16", "uneven": False, "host": False},
        # The headline benchmark: 10k queries on 1M x 768, the graph built on full-dimensional codes,
        # L = rerank = 152 with an expansion budget of 76 (recall@10 of 0.90).
        {"name": "search_batch_1m_768", "kind": "search", "n": 1000000, "D": 768, "d": 160, "bits": 8, "R": 64,
         "L_build": 128, "metric": "ip", "graph": "full", "m": 10000, "k": 10, "L": 152, "rerank": 152, "hops": 76,
         "width": 2, "projection": "bf16", "uneven": False, "host": False},
        # An uneven batch of out-of-distribution queries, per-query k of 1, 10 or 100 and L of 20 to 300
        # (the batching workload's shape, D = 200, d = 64, on 1M rows), no expansion budget.
        {"name": "search_uneven_1m_200", "kind": "search", "n": 1000000, "D": 200, "d": 64, "bits": 8, "R": 64,
         "L_build": 128, "metric": "ip", "graph": "primary", "m": 50000, "k": 100, "L": 300, "rerank": 300, "hops": 0,
         "width": 2, "projection": "fp32", "uneven": True, "host": False},
        # Queries and results in host memory, LVQ-4 primaries and the e4m3 projection (the precision
        # workload's options): a front end that hands over pinned batches.
        {"name": "search_host_lvq4_300k", "kind": "search", "n": 300000, "D": 768, "d": 160, "bits": 4, "R": 64,
         "L_build": 128, "metric": "ip", "graph": "primary", "m": 20000, "k": 10, "L": 256, "rerank": 256, "hops": 256,
         "width": 2, "projection": "fp8", "uneven": False, "host": True},
        # Euclidean search (the gist-like workload: D = 960, not normalised, L2 metric), 3000 queries.
        {"name": "search_l2_200k_960", "kind": "search", "n": 200000, "D": 960, "d": 160, "bits": 8, "R": 64,
         "L_build": 128, "metric": "l2", "graph": "primary", "m": 3000, "k": 10, "L": 72, "rerank": 72, "hops": 72,
         "width": 2, "projection": "bf16", "uneven": False, "host": False},
        # Building the graph on reduced primaries (the paper's fast construction), batch of the tests
        # at scale.
        {"name": "build_primary_200k_160", "kind": "build", "n": 200000, "d": 160, "bits": 8, "R": 64, "L_build": 128,
         "alpha": 1.02, "batch": 65536, "rule": 1},
        # Building on LVQ-8 codes of the unreduced vectors (the graph that the searches share).
        {"name": "build_full_50k_768", "kind": "build", "n": 50000, "d": 768, "bits": 8, "R": 64, "L_build": 128,
         "alpha": 1.02, "batch": 16384, "rule": 1},
        # Encoding a database for the headline workload, and a small one where the call's fixed costs count.
        {"name": "encode_1m_768", "kind": "encode", "n": 1000000, "D": 768, "d": 160, "bits": 8, "sbits": 8,
         "projection": "bf16"},
        {"name": "encode_10k_128", "kind": "encode", "n": 10000, "D": 128, "d": 32, "bits": 8, "sbits": 8,
         "projection": "fp32"},
        # Learning LeanVec-ID on the benchmark's 100k-row sample.
        {"name": "fit_id_100k_768", "kind": "fit_id", "n": 100000, "D": 768, "d": 160, "projection": "bf16"},
        # One step of the gradient optimiser of LeanVec-OOD: pair loss forward and backward over 10k x
        # 100k pairs, a gradient step, the projection onto the spectral-norm ball.
        {"name": "ood_step_10k_100k_512", "kind": "ood_step", "n": 100000, "m": 10000, "D": 512, "d": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "search", "build", "encode", "fit_id", "ood_step"])
    if kind == "search":
        D = rng.choice([96, 100, 128, 200, 256, 300, 384, 512, 768, 960, rng.randint(80, 960)])
        bits = rng.choice([8, 8, 4])
        d = min(D, rng.choice([32, 64, 96, 128, 160, 192, rng.randint(24, 224)]))
        m = _log(rng, 1, 20000)
        L = rng.randint(20, 300)
        hops = rng.choice([0, (L + 1) // 2, L])
        uneven = rng.random() < 0.25
        k = rng.choice([1, 10, 10, 100]) if not uneven else 100
        L = max(L, k)
        projection = rng.choice(["fp32", "bf16", "fp8", "tf32x3"])
        if projection == "tf32x3" and D % 4:
            projection = "fp32"
        n = min(_log(rng, 10000, 1000000), 400_000_000 // D)
        return {"kind": kind, "n": n, "D": D, "d": d, "bits": bits, "R": rng.choice([32, 64]), "L_build": 64,
                "metric": rng.choice(["ip", "ip", "l2"]), "graph": "primary", "m": m, "k": k, "L": L,
                "rerank": rng.choice([L, L, max(k, L // 2)]), "hops": hops, "width": rng.choice([1, 2, 2]),
                "projection": projection, "uneven": uneven, "host": rng.random() < 0.25}
    if kind == "build":
        full = rng.random() < 0.3
        return {"kind": kind, "n": _log(rng, 2000, 50000 if full else 200000),
                "d": rng.randint(300, 960) if full else rng.choice([32, 64, 128, 160, rng.randint(24, 224)]),
                "bits": 8 if full else rng.choice([8, 8, 4]), "R": rng.choice([32, 48, 64]),
                "L_build": rng.choice([64, 100, 128]), "alpha": rng.choice([0.95, 1.0, 1.02]),
                "batch": rng.choice([1024, 4096, 16384, 65536]), "rule": rng.choice([0, 1])}
    if kind == "encode":
        D = rng.choice([96, 128, 200, 256, 512, 768, 960, rng.randint(80, 960)])
        n = min(_log(rng, 1000, 1000000), 768_000_000 // D)
        projection = rng.choice(["fp32", "bf16", "fp8"])
        return {"kind": kind, "n": min(n, 200000) if projection == "fp32" else n, "D": D,
                "d": min(D, rng.choice([32, 64, 128, 160, rng.randint(24, 240)])), "bits": rng.choice([8, 8, 4]),
                "sbits": rng.choice([8, 8, 16]), "projection": projection}
    if kind == "fit_id":
        D = rng.choice([96, 128, 200, 256, 512, 768, rng.randint(64, 768)])
        return {"kind": kind, "n": _log(rng, 2000, 100000), "D": D, "d": max(8, int(D * rng.uniform(0.12, 0.4))),
                "projection": rng.choice(["bf16", "fp32"])}
    D = rng.choice([128, 200, 256, 384, 512])
    return {"kind": kind, "n": _log(rng, 2000, 100000), "m": _log(rng, 500, 10000), "D": D,
            "d": min(D // 2, rng.choice([16, 32, 64, 96, 128]))}


# ----------------------------------------------------------------------------- inputs
def _gen(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed((seed * 1000003 + stream) & 0x7FFFFFFFFFFF)
    return g


def _basis(D: int, g: torch.Generator) -> torch.Tensor:
    """A random orthogonal D x D matrix, columns = principal axes."""
    q, r = torch.linalg.qr(torch.randn(D, D, generator=g, device="cuda"))
    return (q * torch.sign(torch.diagonal(r))[None, :]).contiguous()


def _spectrum(D: int) -> torch.Tensor:
    s = 1.0 / torch.arange(1, D + 1, dtype=torch.float64, device="cuda")
    return torch.sqrt(s * (D / s.sum())).float()


def _rows(n, means, basis, sq, g, unit, chunk=131072):
    """n draws of the mixture: mean of a random component + 0.3 x noise with the spectrum sq^2 in `basis`."""
    C, D = means.shape
    out = torch.empty(n, D, device="cuda")
    bt = basis.T.contiguous()
    for s in range(0, n, chunk):
        e = min(n, s + chunk)
        c = torch.randint(0, C, (e - s,), generator=g, device="cuda")
        x = means[c] + 0.3 * ((torch.randn(e - s, D, generator=g, device="cuda") * sq) @ bt)
        out[s:e] = x / x.norm(dim=1, keepdim=True).clamp_min(1e-30) if unit else x
    return out


def _mixture(D, seed):
    g = _gen(seed, 1)
    U, sq = _basis(D, g), _spectrum(D)
    means = (torch.randn(COMPONENTS, D, generator=g, device="cuda") * sq) @ U.T.contiguous()
    return means, U, sq


def _shifted(means, U, seed):
    """Query mixture of the out-of-distribution workloads: a global gap, an offset per component and
    the noise in a rotated basis."""
    g = _gen(seed, 2)
    C, D = means.shape
    gap = 0.5 * torch.randn(D, generator=g, device="cuda")
    off = 0.25 * torch.randn(C, D, generator=g, device="cuda")
    return means + gap + off, (U @ _basis(D, g)).contiguous()


def _mean(X):
    return X.mean(dim=0, dtype=torch.float64).float()


class _State:
    pass


def _prepare_search(case, seed):
    D, d, n, m = case["D"], case["d"], case["n"], case["m"]
    l2 = case["metric"] == "l2"
    means, U, sq = _mixture(D, seed)
    X = _rows(n, means, U, sq, _gen(seed, 3), unit=not l2)
    if case["uneven"]:
        qmeans, qbasis = _shifted(means, U, seed)
    else:
        qmeans, qbasis = means, U
    Q = _rows(m, qmeans, qbasis, sq, _gen(seed, 4), unit=not l2)
    st = _State()
    st.A = U[:, :d].T.contiguous()  # the distribution's leading principal axes
    Y = X @ st.A.T
    idx = lv.Index(metric=lv.METRIC_L2 if l2 else lv.METRIC_IP)
    idx.set_primary(Y, _mean(Y), case["bits"], D)
    idx.set_secondary(X, _mean(X))
    alpha, rule = (1.2, lv.PRUNE_SCALED) if l2 else (1.02, lv.PRUNE_UNIT_L2)
    if case["graph"] == "full":
        gi = lv.Index(metric=lv.METRIC_L2 if l2 else lv.METRIC_IP).set_primary(X, _mean(X), 8, D)
        gi.build_graph(R=case["R"], L_build=case["L_build"], alpha=alpha, passes=2, batch=65536, rule=rule)
        adj, entry = gi.get_graph()
        gi.close()
        idx.set_graph(adj, entry)
    else:
        idx.build_graph(R=case["R"], L_build=case["L_build"], alpha=alpha, passes=2, batch=16384, rule=rule)
    st.idx = idx
    st.kw = dict(k=case["k"], L=case["L"], rerank=case["rerank"], max_hops=case["hops"], width=case["width"],
                 projection=PREC[case["projection"]])
    if case["uneven"]:
        g = _gen(seed, 5)
        ks = torch.tensor([1, 10, case["k"]], device="cuda")[torch.randint(0, 3, (m,), generator=g, device="cuda")]
        Ls = torch.maximum(torch.randint(20, case["L"] + 1, (m,), generator=g, device="cuda"), ks)
        rr = torch.clamp(Ls, max=case["rerank"])
        desc = torch.stack([ks, Ls, torch.maximum(rr, ks), torch.full_like(ks, case["hops"])], dim=1).to(torch.int32)
        st.kw["desc"] = desc.cpu() if case["host"] else desc.contiguous()
    st.host = case["host"]
    if st.host:
        st.Q = Q.cpu().pin_memory()
        st.kw["batch"] = max(1, (m + 1) // 2)
        st.kw["out"] = (torch.empty((m, case["k"]), dtype=torch.int32).pin_memory(),
                        torch.empty((m, case["k"]), dtype=torch.float32).pin_memory())
    else:
        st.Q = Q
    return st


def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        st = _prepare_search(case, seed)
    else:
        st = _State()
        st.seed = seed
        D = case["d"] if kind == "build" else case["D"]
        means, U, sq = _mixture(D, seed)
        X = _rows(case["n"], means, U, sq, _gen(seed, 3), unit=True)
        if kind == "build":
            st.idx = lv.Index().set_primary(X, _mean(X), case["bits"], D)
            st.kw = dict(R=case["R"], L_build=case["L_build"], alpha=case["alpha"], passes=2,
                         batch=min(case["batch"], case["n"]), rule=case["rule"])
        elif kind == "encode":
            st.X, st.B, st.idx = X, U[:, :case["d"]].T.contiguous(), lv.Index()
            st.kw = dict(primary_bits=case["bits"], secondary_bits=case["sbits"], precision=PREC[case["projection"]])
        elif kind == "fit_id":
            st.X, st.d, st.precision = X, case["d"], PREC[case["projection"]]
        else:
            qmeans, qbasis = _shifted(means, U, seed)
            st.X, st.Q = X, _rows(case["m"], qmeans, qbasis, sq, _gen(seed, 4), unit=True)
            st.A, st.B = _start(case, U, seed)
    st.kind = kind
    return st


def _start(case, U, seed):
    """An iterate of the optimiser: the principal axes, scaled and perturbed a little, so that some
    singular values lie above 1 and some below."""
    g = _gen(seed, 6)
    P = U[:, :case["d"]].T
    out = []
    for _ in range(2):
        s = 0.9 + 0.2 * torch.rand(case["d"], 1, generator=g, device="cuda")
        out.append((P * s + 0.002 * torch.randn(P.shape, generator=g, device="cuda")).contiguous())
    return out


STEP = 0.05  # the optimiser's step in ood_step


def run(st):
    if st.kind == "search":
        if st.host:
            return st.idx.search_host(st.Q, st.A, **st.kw)
        return st.idx.search(st.Q, st.A, **st.kw)
    if st.kind == "build":
        st.idx.build_graph(**st.kw)
        return st.idx.get_graph()
    if st.kind == "encode":
        st.idx.encode(st.X, st.B, **st.kw)
        return {"primary": st.idx.primary_records(), "primary_mean": st.idx.primary_mean(),
                "secondary": st.idx.secondary_records()}
    if st.kind == "fit_id":
        return lv.leanvec_fit_id(st.X, st.d, precision=st.precision)
    A, B = st.A.clone().requires_grad_(True), st.B.clone().requires_grad_(True)
    loss = lv.OODLoss.apply(A, B, st.Q, st.X)
    loss.backward()
    with torch.no_grad():
        A2 = lv.leanvec_spectral_clip(A - STEP * A.grad)
        B2 = lv.leanvec_spectral_clip(B - STEP * B.grad)
    return {"loss": loss.detach(), "gA": A.grad, "gB": B.grad, "A": A2, "B": B2}


# ------------------------------------------------------------------- floors and exact values
def _stride(dim, bits, l2=False):
    code = (dim if bits == 8 else (dim + 1) // 2 if bits == 4 else 2 * dim)
    if bits == 16:
        return (code + 31) // 32 * 32
    return ((code + 15) // 16 * 16 + (32 if l2 else 16) + 31) // 32 * 32


def work(case):
    kind = case["kind"]
    if kind == "search":
        # per query: the query, the adjacency rows of its expansions, about 12 newly met primaries per
        # expansion, the reranked secondaries and the results; a store is read once at most
        m, n, D, d, k = case["m"], case["n"], case["D"], case["d"], case["k"]
        L = 0.5 * (20 + case["L"]) if case["uneven"] else case["L"]
        r = 0.5 * (20 + case["rerank"]) if case["uneven"] else case["rerank"]
        hops = case["hops"] or L
        l2 = case["metric"] == "l2"
        scored = 12.0 * hops
        data = (min(m * hops, n) * 4 * case["R"] + min(m * scored, n) * _stride(d, case["bits"], l2) +
                min(m * r, n) * _stride(D, 8, l2))
        return {"bytes": m * 4 * D + 4 * d * D + data + m * 8 * k, "flops": 2.0 * m * (D * d + scored * d + r * D)}
    if kind == "build":
        # two passes of a beam search per node (about 12 new records in each of L_build expansions) and
        # the pair scores of the pruning (a pool of L_build + R against R kept)
        n, d, R, Lb = case["n"], case["d"], case["R"], case["L_build"]
        pairs = 2.0 * n * (min(12.0 * Lb, n) + (Lb + R) * R / 2)
        return {"bytes": n * _stride(d, case["bits"]) + n * 4.0 * R, "flops": 2.0 * d * pairs}
    if kind == "encode":
        n, D, d = case["n"], case["D"], case["d"]
        return {"bytes": 4.0 * n * D + 4.0 * d * D + n * (_stride(d, case["bits"]) + _stride(D, case["sbits"])),
                "flops": 2.0 * n * D * d + 10.0 * n * (D + d)}
    if kind == "fit_id":
        n, D, d = case["n"], case["D"], case["d"]
        return {"bytes": 4.0 * n * D + 4.0 * d * D, "flops": 1.0 * n * D * (D + 1) + 4 / 3 * D ** 3 + 4.0 * D * D * d}
    n, m, D, d = case["n"], case["m"], case["D"], case["d"]
    # residuals of all pairs once forward and once backward, their two contractions, two clips
    return {"bytes": 4.0 * (n + m) * D + 16.0 * d * D, "flops": 2.0 * n * m * (2 * D + 2 * d) + 20.0 * d * d * D}


def exact(case, seed):
    kind = case["kind"]
    if kind == "encode":
        # The records are bytes; the mean is a computed number.  It follows the rounding of the
        # projection's operands, which is the caller's choice: only the float32 one is given.
        if case["projection"] != "fp32":
            return None
        st = prepare(case, seed)
        mean = torch.zeros(case["d"], dtype=torch.float64, device="cuda")
        for c in st.X.split(131072):
            mean += (c.double() @ st.B.double().T).sum(dim=0)
        return {"primary": None, "primary_mean": (mean / case["n"]).cpu(), "secondary": None}
    if kind == "fit_id":
        # the leading eigenvectors of the second moment of the rows in the precision asked for
        st = prepare(case, seed)
        K = torch.zeros(case["D"], case["D"], dtype=torch.float64, device="cuda")
        for c in st.X.split(65536):
            c = (c.bfloat16() if case["projection"] == "bf16" else c).double()
            K += c.T @ c
        w, V = np.linalg.eigh(K.cpu().numpy())
        P = V[:, ::-1][:, :case["d"]].T
        j = np.argmax(np.abs(P), axis=1)
        return np.ascontiguousarray(P * np.where(P[np.arange(P.shape[0]), j] < 0, -1.0, 1.0)[:, None])
    if kind == "ood_step":
        # the pair loss and its gradients through the second moments, then the clipped singular values
        st = prepare(case, seed)
        A, B, nm = st.A.double(), st.B.double(), float(case["n"]) * case["m"]
        KQ = st.Q.double().T @ st.Q.double()
        KX = torch.zeros_like(KQ)
        for c in st.X.split(65536):
            KX += c.double().T @ c.double()
        AK, BK = A @ KQ, B @ KX
        loss = (((AK @ A.T) * (BK @ B.T).T).sum() + (KQ * KX).sum() - 2.0 * (AK * BK).sum()) / nm
        gA = 2.0 * ((BK @ B.T) @ AK - BK @ KQ) / nm
        gB = 2.0 * ((AK @ A.T) @ BK - AK @ KX) / nm

        def clip(M):
            u, s, vt = np.linalg.svd(M.cpu().numpy(), full_matrices=False)
            return (u * np.minimum(s, 1.0)) @ vt

        return {"loss": loss.cpu(), "gA": gA.cpu(), "gB": gB.cpu(), "A": clip(A - STEP * gA), "B": clip(B - STEP * gB)}
    return None  # ids of a walk over the built graph and its adjacency: whole numbers, compared as they are
