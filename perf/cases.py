"""The measured work of this library: graph builds, batched and single searches, learned-stop
training and exact k-NN, through the public calls of paper_2510_05975_gb300.cng, on the data
shapes of paper_2510_05975_gb300.synth (drawn on the GPU here, from the seed alone).

listed() and draw() give cases, prepare() what a program holds before the call, run() one call,
work() the bytes and operations the call cannot do without, exact() its 64-bit values where the
outputs have values that do not depend on a graph.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_05975_gb300 import cng

LATENT = 16  # dimension of the subspace that the descriptor-like mixtures share


def _build(name, data, n, d, L, R, alpha, **more):
    return dict(name=name, kind="build", data=data, n=n, d=d, L=L, R=R, alpha=alpha, **more)


def _search(name, data, n, d, L, R, alpha, nq, k, beam, **more):
    return dict(name=name, kind="search", data=data, n=n, d=d, L=L, R=R, alpha=alpha, nq=nq, k=k,
                beam=beam, **more)


def listed():
    return [
        # a small collection indexed on the fly (a session's embeddings, a unit of a larger job):
        # launches, host steps and the phases' fixed costs count
        _build("build_gauss10k", "gauss", 10_000, 32, 64, 32, 1.2),
        # the headline build: 1M byte-valued descriptors stored as FP32
        _build("build_sift1m", "sift", 1_000_000, 128, 128, 32, 1.2),
        # unit-normalised embeddings under inner product, a wider graph and longer lists
        _build("build_deep1m", "deep", 1_000_000, 96, 160, 48, 1.3, ip=True),
        # wide rows of high intrinsic dimension (odd count): K-streamed screen, hub merges and a
        # connectivity phase with many unreached points
        _build("build_gist", "gist", 50_003, 960, 128, 32, 1.2, slots=32, connect=128),
        # FP16 storage, a count that fills no tile
        _build("build_bigann_f16", "bigann", 999_983, 128, 128, 32, 1.2, half=True),
        # batched serving of byte-valued descriptors from device buffers, one captured graph
        _search("search_sift_10k", "sift", 1_000_000, 128, 128, 32, 1.2, 10_000, 10, 36, graph=True),
        # batched serving of FP32 embeddings (general kernel, FP64 near-ties)
        _search("search_deep_10k", "deep", 1_000_000, 96, 160, 48, 1.3, 10_000, 10, 24, ip=True),
        # a large uneven batch on FP16 rows
        _search("search_bigann_100k", "bigann", 999_983, 128, 128, 32, 1.2, 100_000, 10, 64, half=True),
        # the learned early stop where it is meant to pay: wide beams for a high recall
        _search("search_learned_f16", "bigann", 500_009, 128, 128, 32, 1.2, 10_000, 10, 192,
                half=True, learned=True),
        # one query from host memory to host memory: the latency of an interactive request
        _search("search_one", "sift", 100_003, 128, 128, 32, 1.2, 1, 10, 36, host=True),
        # fitting the stop network: traced searches, then its training steps
        dict(name="stop_train", kind="train", data="sift", n=250_000, d=128, L=128, R=32, alpha=1.2,
             nq=10_000, k=10, beam=36),
        # ground truth for recall: exact neighbours of held-out queries
        dict(name="knn_10k", kind="knn", data="sift", n=1_000_000, d=128, m=10_000, k=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    data = rng.choice(["gauss", "sift", "sift", "deep", "gist", "bigann"])
    n = _log(rng, *{"gauss": (2_000, 60_000), "gist": (2_000, 30_000)}.get(data, (5_000, 400_000)))
    d = {"gauss": rng.randint(12, 40), "sift": rng.choice([64, 100, 128, 128]), "deep": rng.randint(48, 160),
         "gist": rng.randint(300, 960), "bigann": rng.choice([96, 128])}[data]
    L = rng.choice([48, 64, 100, 128, 160, 200])
    case = dict(kind=rng.choice(["build", "build", "search", "search", "knn", "train"]), data=data, n=n, d=d)
    if case["kind"] == "knn":
        case["m"] = _log(rng, 8, 20_000)
        case["k"] = rng.choice([1, 10, 33, 100, 128, 200])
        return case
    case.update(L=L, R=rng.choice([16, 24, 32, 48]), alpha=rng.choice([1.1, 1.2, 1.3]))
    if data == "deep":
        case["ip"] = True
    if data == "bigann":
        case["half"] = rng.random() < 0.7
    if data == "gist":
        case.update(slots=32, connect=128)
    if case["kind"] == "build":
        if rng.random() < 0.25:
            case["adaptive"] = True
        return case
    case["k"] = rng.choice([1, 10, 10, 20])
    if case["kind"] == "train":
        case.update(nq=_log(rng, 500, 8_000), beam=rng.randint(24, 64))
        return case
    case.update(nq=_log(rng, 1, 40_000), beam=_log(rng, 20, 256))
    if data == "gist":
        case["nq"] = min(case["nq"], 2_000)
    option = rng.choice(["graph", "host", "learned", "none"])
    if option != "none":
        case[option] = True
    return case


# ---- inputs ------------------------------------------------------------------------------------


class _Data:
    """One collection: base and query rows of the same mixture."""

    def __init__(self, case, seed):
        self.case, self.d = case, case["d"]
        self.gen = torch.Generator(device="cuda").manual_seed(seed * 16 + 3)
        d, kind = self.d, case["data"]
        if kind in ("sift", "deep", "bigann"):
            spread = {"sift": 25.0 / 4, "deep": 0.5 / math.sqrt(LATENT * d), "bigann": 0.5 / 4}[kind]
            centres = {"sift": 64, "deep": 256, "bigann": 1024}[kind]
            if kind == "sift":
                self.c0 = torch.randint(112, 144, (d,), generator=self.gen, device="cuda").float()
            elif kind == "deep":
                g = self._normal(d)
                self.c0 = g / g.norm()
            else:
                self.c0 = torch.zeros(d, device="cuda")
            self.load = self._normal(d, LATENT) * spread
            self.centre = self._normal(centres, LATENT)
        elif kind == "gist":
            self.c0 = 0.1 * self._normal(100, d)
            u = torch.rand((100, d), generator=self.gen, device="cuda")
            self.scale = (0.5 * math.log(0.01) * u).exp()  # variances log-uniform on [0.01, 1]

    def _normal(self, *shape):
        return torch.randn(shape, generator=self.gen, device="cuda")

    def rows(self, m):
        kind, d = self.case["data"], self.d
        if kind == "gauss":
            x = self._normal(m, d)
        elif kind == "gist":
            a = torch.randint(0, 100, (m,), generator=self.gen, device="cuda")
            x = self.c0[a] + self.scale[a] * self._normal(m, d)
        else:
            a = torch.randint(0, len(self.centre), (m,), generator=self.gen, device="cuda")
            z = self.centre[a] + self._normal(m, LATENT)
            noise = {"sift": 2.0, "deep": 0.05 / math.sqrt(d), "bigann": 0.05}[kind]
            x = self.c0 + (z[:, :, None] * self.load.t()[None]).sum(1) if m <= 256 else \
                self.c0 + z @ self.load.t()
            x = x + noise * self._normal(m, d)
            if kind == "sift":
                x = x.clamp(0, 255).round()
            elif kind == "deep":
                x = x / x.norm(dim=1, keepdim=True)
        return x.half() if self.case.get("half") else x


def _build_args(case):
    args = dict(alpha=case["alpha"], R=case["R"], L=case["L"], connect_L=case.get("connect", 0),
                repair_slots=case.get("slots", 0))
    if case.get("ip"):
        args["metric"] = cng.CNG_IP_AS_L2
    if case.get("adaptive"):
        args["adaptive"] = (0.9, 1.6, 0.05)
    return args


def prepare(case, seed):
    data = _Data(case, seed)
    kind = case["kind"]
    points = data.rows(case["n"])
    if kind == "build":
        return dict(case=case, points=points, args=_build_args(case))
    if kind == "knn":
        return dict(case=case, points=points, rows=data.rows(case["m"]))
    queries = data.rows(case["nq"]).float()
    index, _ = cng.cng_build(points, **_build_args(case))
    state = dict(case=case, index=index, queries=queries, model=None)
    if case.get("learned"):
        train = data.rows(2_000).float()
        state["model"], _ = cng.cng_stop_train(index, train, k=case["k"], L=case["beam"])
    if kind == "search":
        nq, k = case["nq"], case["k"]
        shapes = dict(ids=((nq, k), torch.int32), dists=((nq, k), torch.float32), hops=((nq,), torch.int32))
        if case.get("host"):
            state["queries"] = queries.cpu().numpy()
            as_numpy = {torch.int32: np.int32, torch.float32: np.float32}
            state["out"] = {key: np.empty(s, as_numpy[t]) for key, (s, t) in shapes.items()}
        else:
            state["out"] = {key: torch.empty(s, dtype=t, device="cuda") for key, (s, t) in shapes.items()}
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "build":
        index, _ = cng.cng_build(state["points"], **state["args"])
        adj, deg, _, entry = cng.cng_graph(index)
        out = dict(adj=adj.clone(), deg=deg.clone(), entry=entry)  # the index is freed here
        cng.cng_free(index)
        return out
    if kind == "knn":
        ids, dists, _ = cng.cng_knn(state["points"].float(), case["k"], rows=state["rows"].float())
        return dict(ids=ids, dists=dists)
    if kind == "train":
        model, _ = cng.cng_stop_train(state["index"], state["queries"], k=case["k"], L=case["beam"])
        params, mu, sigma, rounded = cng.cng_stop_export(model)
        cng.cng_stop_free(model)
        return dict(params=params, mu=mu, sigma=sigma, rounded=rounded)
    how = dict(mode=cng.CNG_SEARCH_LEARNED, model=state["model"], threshold=0.95, check_every=4,
               min_stable=6) if case.get("learned") else {}
    out = cng.cng_search(state["index"], state["queries"], k=case["k"], L=case["beam"],
                         use_graph=bool(case.get("graph")), out=state["out"], with_stats=False, **how)
    return dict(ids=out["ids"], dists=out["dists"], hops=out["hops"])


def work(case):
    """Points and queries read once, results written once.  Builds: every unordered pair of
    points has one inner product (2 d operations).  Searches: each query explores at least the
    `beam` vertices of its final queue, so it reads their adjacency rows and vectors and takes
    their distances (3 d operations each)."""
    kind, n, d = case["kind"], case["n"], case["d"]
    size = 2 if case.get("half") else 4
    if kind == "build":
        stride = case["R"] + (case.get("slots") or 8)
        return dict(bytes=n * d * size + n * (stride + 1) * 4, flops=float(n) * (n - 1) * d)
    if kind == "knn":
        m, k = case["m"], case["k"]
        return dict(bytes=(n + m) * d * 4 + m * k * 8, flops=2.0 * m * n * d)
    nq, beam = case["nq"], case["beam"]
    row = 1 if case["data"] == "sift" else size  # byte-valued rows need one byte a coordinate
    walk = nq * beam * (case["R"] * 4 + d * row)
    io = nq * d * 4 + (4 * 5313 if kind == "train" else nq * (case["k"] * 8 + 4))
    flops = 3.0 * nq * beam * d
    if kind == "train":  # 4 epochs of forward and backward over each traced hop (at least `beam`)
        flops += 4.0 * nq * beam * 6 * (16 * 64 + 64 * 64 + 64)
    return dict(bytes=walk + io, flops=flops)


def exact(case, seed):
    """Exact neighbours by (distance, id) for k-NN calls; everything else depends on a graph and
    has no value of its own here."""
    if case["kind"] != "knn":
        return None
    data = _Data(case, seed)
    base = data.rows(case["n"]).double()
    rows = data.rows(case["m"]).double()
    k, n = case["k"], case["n"]
    take = min(n, k + 28)
    norm = (base * base).sum(1)
    ids, dists = [], []
    for part in rows.split(max(1, (1 << 28) // n)):
        near = torch.addmm(norm[None], part, base.t(), alpha=-2.0).topk(take, dim=1, largest=False).indices
        near = near.sort(dim=1).values  # by id first: the sort by distance below is stable
        dist = torch.stack([(base[i] - x).square().sum(1) for i, x in zip(near, part)]).sqrt()
        order = dist.sort(dim=1, stable=True)
        ids.append(near.gather(1, order.indices)[:, :k].int())
        dists.append(order.values[:, :k])
    return dict(ids=torch.cat(ids), dists=torch.cat(dists))
