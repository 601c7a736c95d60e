"""Documents on CTAs above 8,192 topics: every topic, count and counter equal to
the oracle's, over rows and columns, in the corpus pass, fold-in, serving and
batches."""
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


def corpus(rng, lengths, V, a):
    off = np.zeros(len(lengths) + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    p = (1.0 + np.arange(V)) ** -a
    return rng.choice(V, size=int(off[-1]), p=p / p.sum()).astype(np.int32), off


LENGTHS = [0, 1, 2, 3, 4, 31, 32, 33, 63, 64, 65, 96, 97, 255, 300, 2600, 400, 4000] + [380] * 60


# the last K of the chain kernel, the first of this one; C = 17 (five chunks a warp, two for the last), 18, 24, 32
@pytest.mark.parametrize("K", [8192, 8193, 8704, 8705, 12000, 16384])
def test_lockstep(K):
    """The frequent words' columns are longer than the column limit, the others'
    shorter; counts pass one plane and come back."""
    rng = np.random.default_rng(K)
    w, off = corpus(rng, LENGTHS, 40, 1.1)
    w[off[15]:off[16]:2] = 3
    alpha = rng.uniform(0.01, 0.05, K).astype(np.float32)
    alpha[[0, 17, K - 1]] = 60.0
    s, ch = lockstep(w, off, K, 40, alpha, 0.01, seed=K, sweeps=3, check_counts_every=3, coop_min_len=1)
    n_w = np.diff(s.word_tables()["col_ptr"])
    assert n_w.max() > 512 and n_w.min() <= 512, n_w
    assert not first_mismatch(s.infer(w, off, 3, seed=4), O.infer(ch.tables, w, off, 3, 4), off)
    for slice_tokens in (0, 33):
        srv = P_server(s, slice_tokens)
        docs = {d: w[off[d]:off[d + 1]] for d in range(20) if LENGTHS[d]}
        for d, words in docs.items():
            srv.submit(d, d, words, 3)
        got = {}
        while len(got) < len(docs):
            for r in srv.poll(timeout_ms=500):
                assert r["status"] == 0
                got[r["req_id"]] = r["z"]
        srv.close()
        for d, words in docs.items():
            assert np.array_equal(got[d], O.infer(ch.tables, words, np.array([0, len(words)]), 3, d)), (slice_tokens, d)
    s.close()


def P_server(s, slice_tokens):
    import paper_1704_03581_gb300 as P
    return P.Server(s, token_budget=20000, max_slots=32, slice_tokens=slice_tokens)


def test_batch_of_every_form():
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(8)
    chains = []
    for i, K in enumerate([60, 200, 400, 700, 3000, 8192, 8193, 10000]):
        w, off = corpus(rng, np.append(rng.integers(20, 200, size=40), [700, 900]), 60, 0.8)
        chains.append(dict(w=w, doc_off=off, K=K, V=60, alpha=0.05, beta=0.01, seed=20 + i))
    b = P.Batch(chains, coop_min_len=150)
    b.sweep(3)
    for i, c in enumerate(chains):
        one = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], 0.05, 0.01, c["seed"], coop_min_len=-1).sweep(3)
        assert np.array_equal(b.z(i), one.z()), c["K"]
        one.close()
    b.close()
