"""The Phi-step's passes at the edges of their ways, against the oracle: every
count, table entry and topic equal."""
import numpy as np
import pytest

from parity_util import lockstep

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03581_gb300 import build
    build.build()


def corpus_of(rng, sizes, docs):
    """Word v occurs sizes[v] times; the tokens, shuffled, in `docs` documents."""
    w = rng.permutation(np.repeat(np.arange(len(sizes), dtype=np.int32), sizes))
    return w, np.linspace(0, w.size, docs + 1).astype(np.int64)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("K", [1, 31, 33, 1000, 4096, 4097])
def test_word_counts_by_warps_ctas_and_chunks(K, mode):
    """More words than one wave of CTAs, so that words of up to 256 tokens go
    to warps (K <= 4096): sizes around a warp's loads, that limit and the
    limit of the words that several CTAs histogram (4,096 in a small corpus)."""
    rng = np.random.default_rng(K)
    sizes = np.full(2600, 1)
    sizes[:24] = [0, 2, 31, 32, 33, 127, 128, 129, 160, 255, 256, 257, 258, 511, 1025, 4095, 4096, 4097, 8192, 8193, 12289, 0, 0, 5]
    w, off = corpus_of(rng, rng.permutation(sizes), 60)
    s, _ = lockstep(w, off, K, 2600, rng.uniform(0.05, 0.5, K).astype(np.float32), 0.02, seed=K, sweeps=2 if K <= 1000 else 1,
                    check_counts_every=1, phi_mode=mode if K <= 1000 else 0)
    s.close()


@pytest.mark.parametrize("V", [2047, 2048, 2049, 4097, 10241])
def test_column_offsets_across_chunks(V):
    """Words around the entries that a CTA of the column scan takes."""
    rng = np.random.default_rng(V)
    w, off = corpus_of(rng, rng.poisson(3, V), 40)
    s, _ = lockstep(w, off, 7, V, np.full(7, 0.1, np.float32), 0.05, seed=3, sweeps=2, check_counts_every=2)
    s.close()


def test_column_offsets_of_larger_chunks():
    """Past 256 CTAs of 2,048 words each a CTA takes more."""
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(1)
    V = 700001
    w = rng.integers(0, V, 300000).astype(np.int32)
    s = P.Sampler(w, np.linspace(0, w.size, 501).astype(np.int64), 5, V, 0.1, 0.02, 1)
    s.phi_step()
    t = s.word_tables()
    assert t["col_ptr"][0] == 0 and t["col_ptr"][-1] == t["topic"].size
    # every column's topics ascend, and a new column starts where they do not
    cuts = np.nonzero(np.diff(t["topic"].astype(np.int64)) <= 0)[0] + 1
    assert np.isin(cuts, t["col_ptr"]).all()
    assert np.array_equal(np.bincount(t["topic"], weights=t["c"], minlength=5).astype(np.int64), t["S"])
    s.close()


def test_batch_counts_of_mixed_chains():
    """One launch's warps take rare words of chains of different K in turn."""
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(8)
    chains = []
    for i, (K, V) in enumerate([(5, 3000), (100, 2500), (1500, 1200), (33, 4000)]):
        w, off = corpus_of(rng, rng.integers(0, 12, V) + (np.arange(V) < 9) * 300, 50)
        chains.append(dict(w=w, doc_off=off, K=K, V=V, alpha=np.full(K, 0.1, np.float32), beta=0.02, seed=i))
    b = P.Batch(chains)
    b.sweep(3)
    for i, c in enumerate(chains):
        s = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], c["alpha"], c["beta"], c["seed"])
        s.sweep(3)
        assert np.array_equal(b.z(i), s.z()), f"chain {i} differs from its single-chain run"
        s.close()
    b.close()


@pytest.mark.parametrize("K", [1, 2, 33, 255, 257, 600])
def test_alias_pairing(K):
    """Full and sparse columns around the 256 slots that pair in shared memory."""
    rng = np.random.default_rng(K)
    sizes = np.concatenate([np.full(8, 4 * K), rng.integers(0, 60, 60)])
    w, off = corpus_of(rng, sizes, 30)
    s, _ = lockstep(w, off, K, sizes.size, rng.uniform(0.001, 5.0, K).astype(np.float32), 0.3, seed=K, sweeps=2)
    s.close()


@pytest.mark.parametrize("K,alpha", [(900, 256.0), (1100, 256.0), (1500, 100.0), (4200, 256.0)])
def test_alias_pairing_past_64_bits(K, alpha):
    """Long columns of even counts under a large alpha: n A passes 2^64 for the
    frequent words, not for the rare ones."""
    rng = np.random.default_rng(K)
    sizes = np.concatenate([np.full(4, 3 * K), rng.integers(0, 9, 40)])
    w, off = corpus_of(rng, sizes, 30)
    s, ch = lockstep(w, off, K, sizes.size, np.full(K, alpha, np.float32), 40.0, seed=K, sweeps=2)
    t = s.word_tables()
    n = np.diff(t["col_ptr"])
    assert any(int(a) * int(c) >= 1 << 64 for a, c in zip(t["A"].view(np.uint64), n))
    s.close()


@pytest.mark.parametrize("K,V", [(1, 1), (31, 255), (256, 256), (257, 257), (512, 272), (513, 40), (1024, 60), (1025, 33), (7, 4400)])
def test_dirichlet_passes(K, V):
    """Row sums across chunks of 256 words and batches of 16, and the
    selection's registers (256, 512, 1,024 topics) and memory form."""
    rng = np.random.default_rng(K + V)
    w, off = corpus_of(rng, rng.poisson(4, V) + (np.arange(V) < 3) * 200, 20)
    s, _ = lockstep(w, off, K, V, rng.uniform(0.05, 0.5, K).astype(np.float32), 0.02, seed=V, sweeps=2, phi_mode=1)
    s.close()


@pytest.mark.parametrize("alpha", [0.1, None])
def test_log_posterior_of_many_and_of_large_documents(alpha):
    """More than 32 documents per warp, counts past both tables, one row of
    the document table (symmetric alpha) or a row per topic."""
    from test_diag_gpu import check
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(4)
    K, V = 3, 30
    off = np.zeros(500004, np.int64)
    np.cumsum(np.concatenate([[20000, 0, 9000], rng.integers(0, 3, 500000)]), out=off[1:])
    w = rng.integers(0, V, int(off[-1])).astype(np.int32)
    al = np.full(K, alpha, np.float32) if alpha else rng.uniform(0.1, 1.0, K).astype(np.float32)
    s = P.Sampler(w, off, K, V, al, 0.02, seed=7)
    s.sweep(1)
    check(s, off, w, K, V, al, 0.02)
    s.close()
