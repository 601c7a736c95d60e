"""Documents of 2^16 tokens or more on CTAs: counts that pass one, two and three
planes within a pass, in the corpus pass, fold-in, serving and batches, against
the oracle or the one-warp kernel's topics."""
import numpy as np
import pytest

from oracle import oracle as O
from parity_util import first_mismatch, lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03581_gb300 import build
    build.build()


def corpus(rng, lengths, V):
    off = np.zeros(len(lengths) + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    return rng.integers(0, V, size=int(off[-1])).astype(np.int32), off


def few_topics(K):
    alpha = np.full(K, 0.01, np.float32)
    alpha[[0, K - 1]] = 200.0
    return alpha


def settled(rng, off, K, V):
    """A chain whose documents are almost all in the first and the last topic,
    the longest with both just short of 2^16 tokens: (sampler, oracle)."""
    import paper_1704_03581_gb300 as P
    w = rng.integers(0, V, size=int(off[-1])).astype(np.int32)
    z = np.where(rng.random(len(w)) < 0.5, 0, K - 1).astype(np.int16)
    other = rng.random(len(w)) < 0.01
    z[other] = rng.integers(0, K, size=int(other.sum()))
    a, b = off[:2]
    z[a:b] = K - 1
    z[rng.permutation(int(b - a))[:int(b - a) // 2 - 5] + a] = 0
    s = P.Sampler(w, off, K, V, few_topics(K), 0.01, seed=K, coop_min_len=1)
    s.set_z(z, 0)
    ch = O.Chain(w, off, K, V, few_topics(K), 0.01, seed=K)
    ch.z = z.copy()
    return s, ch


def one_sweep(s, ch):
    s.phi_step()
    ch.sweep_index += 1
    ch.phi_step(ch.sweep_index)


# every form of the kernels on both sides of 1,024 and of 8,192 topics
@pytest.mark.parametrize("K", [3, 130, 300, 1000, 1030, 8192, 8200, 16384])
def test_lockstep(K):
    """Counts pass 255 (the document of 500 or 640 tokens) and 65,535 (the longest)
    within the passes; beside them one just short of 2^16 tokens."""
    rng = np.random.default_rng(K)
    # above 8,000 topics more tokens leave for the others
    off = np.append(0, np.cumsum([131000, 500, 65535, 65536] if K < 8000 else [132500, 640, 65535, 65536])).astype(np.int64)
    s, ch = settled(rng, off, K, 12)
    low = high = False
    for sweep in (1, 2, 3):
        one_sweep(s, ch)
        s.z_step()
        ch.z, ch.stats = O.z_step(ch.doc_off, ch.w, ch.z, ch.tables, ch.seed, ch.sweep_index)
        msg = first_mismatch(s.z(), ch.z, off)
        assert not msg, f"sweep {sweep}: " + msg
        st = s.stats()
        assert [st[k] for k in ("tokens", "a_branch", "sum_min", "zero_mass", "sum_inter", "docside")] == list(ch.stats[:6])
        low, high = low or s.m()[0].max() > 65535, high or s.m()[1].max() > 255
    assert low and high
    s.close()


@pytest.mark.parametrize("K", [2, 40, 1100, 9000])
def test_fold_in_and_serving(K):
    import torch
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(K)
    s, ch = settled(rng, np.append(0, np.cumsum([131000, 300, 500])).astype(np.int64), K, 12)
    one_sweep(s, ch)
    new, noff = corpus(rng, [140000, 66000, 40, 3000], 12)
    want = O.infer(ch.tables, new, noff, 2, 5)
    assert K > 2 or np.bincount(want[:140000]).max() > 65535
    assert not first_mismatch(s.infer(new, noff, 2, seed=5), want, noff)
    z = torch.empty(len(new), dtype=torch.int16, device="cuda")
    P.pulda_infer_noalloc(s.h, torch.from_numpy(new).cuda(), torch.from_numpy(noff).cuda(), 2, 5, z)
    assert not first_mismatch(z.cpu().numpy(), want, noff)
    srv = P.Server(s, token_budget=1 << 20, max_slots=8, slice_tokens=0)
    docs = {d: new[noff[d]:noff[d + 1]] for d in range(4)}
    for d, words in docs.items():
        srv.submit(d, 10 + d, words, 2)
    got = {}
    while len(got) < len(docs):
        for r in srv.poll(timeout_ms=500):
            assert r["status"] == 0
            got[r["req_id"]] = r["z"]
    srv.close()
    for d, words in docs.items():
        assert np.array_equal(got[d], O.infer(ch.tables, words, np.array([0, len(words)]), 2, 10 + d)), d
    s.close()


@pytest.mark.parametrize("coop", [0, 65000, 100000, -1])
def test_batch(coop):
    """On CTAs, split between CTAs and the one-warp kernel by the threshold, and
    all on the one-warp kernel."""
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(3)
    chains = []
    for i, K in enumerate([60, 400, 1500, 9000]):
        w, off = corpus(rng, np.append(rng.integers(20, 200, size=60), [80000, 65535, 120000]), 30)
        chains.append(dict(w=w, doc_off=off, K=K, V=30, alpha=few_topics(K), beta=0.01, seed=20 + i))
    b = P.Batch(chains, coop_min_len=coop)
    b.sweep(2)
    for i, c in enumerate(chains):
        one = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], c["alpha"], 0.01, c["seed"], coop_min_len=-1).sweep(2)
        two = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], c["alpha"], 0.01, c["seed"], coop_min_len=coop).sweep(2)
        assert np.array_equal(b.z(i), one.z()) and np.array_equal(two.z(), one.z()), c["K"]
        one.close()
        two.close()
    b.close()


def test_batch_across_the_kernels_ranges():
    """Chains on both sides of the line at which documents of 2^16 tokens or more
    take the kernel with four warps on each token: in a batch they share one."""
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(6)
    for Ks in ([1100, 1500, 7000], [1100, 6000]):
        chains = []
        for i, K in enumerate(Ks):
            w, off = corpus(rng, np.append(rng.integers(20, 400, size=40), [70000, 3000]), 30)
            chains.append(dict(w=w, doc_off=off, K=K, V=30, alpha=few_topics(K), beta=0.01, seed=40 + i))
        b = P.Batch(chains, coop_min_len=100)
        b.sweep(2)
        for i, c in enumerate(chains):
            one = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], c["alpha"], 0.01, c["seed"], coop_min_len=-1).sweep(2)
            assert np.array_equal(b.z(i), one.z()), (Ks, c["K"])
            sb, ss = b.stats(i), one.stats()
            for k in ("tokens", "a_branch", "sum_min", "zero_mass", "sum_inter", "docside"):
                assert sb[k] == ss[k], (Ks, c["K"], k)
            one.close()
        b.close()
