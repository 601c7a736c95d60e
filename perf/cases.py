"""The work that users of this sampler have it do, as cases that can be timed
and compared: training sweeps from the tiny corpus to the large one, the two
Phi draws, many topics, fold-in of new documents through each entry point,
batched chains, the serving loop and the log-posterior diagnostic.

Corpora are drawn on the GPU from the LDA generative process the repository's
own synthetic workloads use (theta_d ~ Dir(0.1), phi_k ~ Dir(0.05 V F) with F
a Zipf law over a permutation of the words, lognormal document lengths), and
chains start from the topics that generated them, as one resumed from a
checkpoint would: the state a long run spends its time in.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1704_03581_gb300 as P

ALPHA, BETA = 0.1, 0.01


def listed() -> list[dict]:
    return [
        # the tiny corpus (~100k tokens): a sweep is launches and one token chain per document
        dict(name="train_tiny", kind="train", phi_mode=0, K=20, V=1000, D=1000, mean=100.0, sd=0.1, zipf=0.0),
        # a UCI bag-of-words-sized corpus, 1.9M tokens: long documents, few topics
        dict(name="train_small", kind="train", phi_mode=0, K=100, V=12375, D=1500, mean=1290.0, sd=0.5, zipf=1.0),
        # 12M tokens at K = 1000: the pass and its longest documents weigh about the same
        dict(name="train_mid", kind="train", phi_mode=0, K=1000, V=100000, D=37500, mean=330.0, sd=0.8, zipf=1.05),
        # the headline workload: 99M tokens at K = 1000
        dict(name="train_large", kind="train", phi_mode=0, K=1000, V=100000, D=300000, mean=330.0, sd=0.8, zipf=1.05),
        # a fine-grained topic model: more topics than the document-side bitmaps hold
        dict(name="train_many_topics", kind="train", phi_mode=0, K=3000, V=30000, D=20000, mean=330.0, sd=0.8, zipf=1.05),
        # Algorithm 1's Dirichlet Phi, the sampler the Polya urn is compared with
        dict(name="train_dirichlet", kind="train", phi_mode=1, K=1000, V=50000, D=30000, mean=330.0, sd=0.8, zipf=1.05),
        # eight independent corpora of uneven size and K advanced together, ten sweeps a call
        dict(name="batch_chains", kind="batch", chains=8, Dlo=1000, Dhi=10000, Vlo=5000, Vhi=50000, sweeps=10),
        # one new document folded in from device buffers: a request on its own
        dict(name="fold_in_one", kind="noalloc", K=1000, V=100000, D=20000, docs=1, mean=300.0, sd=0.0, sweeps=50),
        # a batch of new documents already on the GPU, in arrival order
        dict(name="fold_in_device", kind="noalloc", K=1000, V=100000, D=20000, docs=4096, mean=300.0, sd=0.8, sweeps=20),
        # new documents from host memory and their topics back to it
        dict(name="fold_in_host", kind="infer", K=1000, V=100000, D=20000, docs=256, mean=300.0, sd=1.2, sweeps=50),
        # the serving loop: requests submitted together, topics collected as they finish
        dict(name="serve", kind="serve", K=1000, V=100000, D=20000, docs=384, mean=300.0, sd=1.2, sweeps=50),
        # the trace-plot diagnostic of a training run
        dict(name="log_posterior", kind="posterior", K=1000, V=100000, D=37500, mean=330.0, sd=0.8, zipf=1.05),
    ]


def _log(rng, lo, hi) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng) -> dict:
    kind = rng.choice(["train", "train", "train", "train", "dirichlet", "batch", "noalloc", "infer", "serve", "posterior"])
    if kind in ("train", "dirichlet", "posterior"):
        K = int(_log(rng, 10, 3000)) | rng.getrandbits(1)
        V = int(_log(rng, 1000, min(100000, 1.0e8 / K)))
        mean = _log(rng, 50, 1300)
        tokens = _log(rng, 1e5, {"train": 6e6 if K > 2048 else 6e7, "dirichlet": 1e7, "posterior": 1.2e7}[kind])
        return dict(kind="posterior" if kind == "posterior" else "train", phi_mode=int(kind == "dirichlet"), K=K, V=V,
                    D=max(300, int(tokens / mean)), mean=round(mean, 1), sd=round(rng.uniform(0.1, 0.9), 2),
                    zipf=round(rng.uniform(0.9, 1.1), 2))
    if kind == "batch":
        return dict(kind="batch", chains=rng.randint(2, 8), Dlo=500, Dhi=int(_log(rng, 1000, 10000)), Vlo=2000,
                    Vhi=int(_log(rng, 4000, 50000)), sweeps=rng.randint(2, 10))
    K, V = int(_log(rng, 50, 1000)), int(_log(rng, 5000, 100000))
    top = {"noalloc": 4096, "infer": 256, "serve": 384}[kind]
    return dict(kind=kind, K=K, V=V, D=int(_log(rng, 3000, 20000)), docs=int(_log(rng, 1, top)),
                mean=round(_log(rng, 50, 300), 1), sd=round(rng.uniform(0.3, 1.1), 2), sweeps=rng.randint(5, 20))


# ------------------------------------------------------------------ corpora

class _Topics:
    """phi_k ~ Dir(0.05 V F) (or Dir(0.01) when zipf is 0, the tiny corpus),
    kept as the flat cumulative rows that words are looked up in."""

    def __init__(self, seed: int, K: int, V: int, zipf: float):
        self.K, self.V = K, V
        self.gen = torch.Generator(device="cuda").manual_seed(seed)
        if zipf > 0:
            f = (1.0 + torch.randperm(V, generator=self.gen, device="cuda").double()) ** -zipf
            shape = (0.05 * V * f / f.sum()).float()
        else:
            shape = torch.full((V,), 0.01, device="cuda")
        phi = torch._standard_gamma(shape.expand(K, V).contiguous(), generator=self.gen).double()
        cum = torch.cumsum(phi, 1)
        cum /= cum[:, -1:].clone()
        self.cum = (cum + torch.arange(K, device="cuda")[:, None]).view(-1)

    def documents(self, lengths: np.ndarray):
        """(word ids, offsets, topics) of documents of these lengths: int32,
        int64 and int16 tensors on the GPU."""
        K, V = self.K, self.V
        off = np.zeros(len(lengths) + 1, np.int64)
        np.cumsum(lengths, out=off[1:])
        n = torch.from_numpy(np.asarray(lengths, np.int64)).cuda()
        w, z = [], []
        step = max(1, 20_000_000 // K)
        for a in range(0, len(lengths), step):
            b = min(len(lengths), a + step)
            theta = torch._standard_gamma(torch.full((b - a, K), ALPHA, device="cuda"), generator=self.gen).double()
            cum = torch.cumsum(theta, 1)
            cum /= cum[:, -1:].clone()
            row = torch.repeat_interleave(torch.arange(b - a, device="cuda"), n[a:b])
            u = torch.rand(row.numel(), generator=self.gen, device="cuda", dtype=torch.float64)
            cum += torch.arange(b - a, device="cuda")[:, None]
            k = (torch.searchsorted(cum.view(-1), u + row, right=True) - row * K).clamp_(0, K - 1)
            u = torch.rand(row.numel(), generator=self.gen, device="cuda", dtype=torch.float64)
            v = (torch.searchsorted(self.cum, u + k, right=True) - k * V).clamp_(0, V - 1)
            w.append(v.int())
            z.append(k.short())
        return torch.cat(w), torch.from_numpy(off), torch.cat(z)


def _lengths(D: int, mean: float, sd: float, lo: int = 1, hi: int = 20000) -> np.ndarray:
    """Lognormal document lengths: of the case alone, so that a case's outputs
    have one size whatever the seed."""
    x = np.random.default_rng(D).lognormal(math.log(mean) - 0.5 * sd * sd, sd, size=D)
    return np.clip(np.rint(x), lo, hi).astype(np.int64)


_side = None


def _stream() -> int:
    """One stream for every handle, as in a program that runs one chain."""
    global _side
    if _side is None:
        _side = torch.cuda.Stream()
    return _side.cuda_stream


def _chain(case: dict, seed: int, topics: _Topics, sweeps: int) -> P.Sampler:
    """A sampler at the generating topics, advanced by `sweeps` sweeps."""
    w, off, z = topics.documents(_lengths(case["D"], case["mean"], case["sd"]))
    s = P.Sampler(w.cpu().numpy(), off.numpy(), case["K"], case["V"], ALPHA, BETA, seed=seed, stream=_stream(),
                  phi_mode=case.get("phi_mode", 0))
    s.set_z(z.cpu().numpy(), 0)
    if sweeps:
        s.sweep(sweeps).sync()
    return s


class _Requests:
    """A trained model and new documents for it, with the server if asked for."""

    def __init__(self, case: dict, seed: int):
        topics = _Topics(seed, case["K"], case["V"], 1.05)
        self.model = _chain(dict(case, mean=330.0, sd=0.8), seed, topics, 2)
        w, off, _ = topics.documents(_lengths(case["docs"], case["mean"], case["sd"], lo=10))
        self.w_dev, self.off_dev = w, off.cuda()
        self.z_dev = torch.empty(w.numel(), dtype=torch.int16, device="cuda")
        self.w, self.off = w.cpu().numpy(), off.numpy()
        self.words = [self.w[a:b] for a, b in zip(self.off[:-1], self.off[1:])]
        self.server = P.Server(self.model, token_budget=1 << 22, max_slots=4096, slice_tokens=0) if case["kind"] == "serve" else None

    def __del__(self):
        if getattr(self, "server", None) is not None:
            self.server.close()


# -------------------------------------------------------------------- cases

def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind == "train":
        s = _chain(case, seed, _Topics(seed, case["K"], case["V"], case["zipf"]), 2)
        return dict(kind=kind, s=s, z=torch.empty(s.N, dtype=torch.int16, device="cuda"))
    if kind == "posterior":
        return dict(kind=kind, s=_chain(case, seed, _Topics(seed, case["K"], case["V"], case["zipf"]), 0))
    if kind == "batch":
        # the repository's batched workload: D, V and mean length log-uniform, K in {50, 100, 200, 500}
        chains = []
        for c in range(case["chains"]):
            D, V, K, mean = _batch_shape(case, c)
            w, off, _ = _Topics(seed + c, K, V, 1.0).documents(_lengths(D, mean, 0.8))
            chains.append(dict(w=w.cpu().numpy(), doc_off=off.numpy(), K=K, V=V, alpha=ALPHA, beta=BETA, seed=seed + c))
        b = P.Batch(chains, stream=_stream())
        b.sweep(12).sync()              # past the launch tuning
        return dict(kind=kind, b=b, chains=len(chains), sweeps=case["sweeps"])
    return dict(kind=kind, r=_Requests(case, seed), K=case["K"], sweeps=case["sweeps"], seed=seed)


def _batch_shape(case: dict, c: int):
    rng = np.random.default_rng(400 + c)
    ex = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))  # noqa: E731
    return int(ex(case["Dlo"], case["Dhi"])), int(ex(case["Vlo"], case["Vhi"])), int(rng.choice([50, 100, 200, 500])), ex(50, 500)


def run(state: dict):
    kind = state["kind"]
    if kind == "train":
        state["s"].sweep(1)
        return P.pulda_get_z_dev(state["s"].h, state["z"])
    if kind == "posterior":
        return state["s"].log_posterior()
    if kind == "batch":
        state["b"].sweep(state["sweeps"])
        return [state["b"].z(c) for c in range(state["chains"])]
    r = state["r"]
    if kind == "noalloc":
        return P.pulda_infer_noalloc(r.model.h, r.w_dev, r.off_dev, state["sweeps"], state["seed"], r.z_dev)
    if kind == "infer":
        return r.model.infer(r.w, r.off, state["sweeps"], state["seed"])
    z = {i: r.server.submit(i, state["seed"] + i, words, state["sweeps"]) for i, words in enumerate(r.words)}
    left = len(z)
    while left:
        for done in r.server.poll():
            if done["status"] != P.PULDA_OK:
                raise RuntimeError("a request failed")
            left -= 1
    return np.concatenate([z[i] for i in range(len(z))])


def work(case: dict) -> dict:
    """Per token and sweep: its word id and topic read, its topic written, and
    the exact conditional's multiply-adds over the topics its document and its
    word share (about 100 at K = 1000); the diagnostic adds one term a count."""
    if case["kind"] == "batch":
        tokens = sum(_batch_shape(case, c)[0] * _batch_shape(case, c)[3] for c in range(case["chains"]))
        return dict(bytes=8 * tokens * case["sweeps"], flops=2 * 50 * tokens * case["sweeps"])
    if case["kind"] == "posterior":
        tokens = case["D"] * case["mean"]
        return dict(bytes=6 * tokens, flops=2 * tokens)
    if case["kind"] == "train":
        tokens = case["D"] * case["mean"]
    else:
        tokens = case["docs"] * case["mean"] * case["sweeps"]
    return dict(bytes=8 * tokens, flops=2 * min(case["K"], 100) * tokens)


def exact(case: dict, seed: int):
    """The log joint of the generating topics in 64 bits; topics are random
    draws and have no such value."""
    if case["kind"] != "posterior":
        return None
    K, V, D = case["K"], case["V"], case["D"]
    lengths = _lengths(D, case["mean"], case["sd"])
    w, _, z = _Topics(seed, K, V, case["zipf"]).documents(lengths)
    d = torch.repeat_interleave(torch.arange(D, device="cuda"), torch.from_numpy(lengths).cuda())
    alpha, beta = float(np.float32(ALPHA)), float(np.float32(BETA))
    g = lambda x: torch.lgamma(x)  # noqa: E731
    c = lambda x: math.lgamma(x)  # noqa: E731
    n_d = torch.bincount(d, minlength=D)
    m = torch.bincount(d * K + z.long(), minlength=D * K)
    m = m[m > 0]
    doc = D * c(K * alpha) - float(g(K * alpha + n_d.double()).sum()) + float((g(alpha + m.double()) - c(alpha)).sum())
    n_k = torch.bincount(z.long(), minlength=K)
    n = torch.bincount(z.long() * V + w.long(), minlength=K * V)
    n = n[n > 0]
    topic = K * c(V * beta) - float(g(V * beta + n_k.double()).sum()) + float((g(beta + n.double()) - c(beta)).sum())
    return np.array([doc + topic, doc, topic])
