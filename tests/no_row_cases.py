"""Cases run against a build whose dense rows are limited to 24 KB
(test_no_rows_gpu.py, PULDA_LIB pointing at it), so that most words are summed
over their columns and groups of tokens mix both kinds: the one-warp, pair and
CTA kernels, fold-in, the server and the batched form, topics, counts and
counters against the oracle or the single-chain run."""
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import paper_1704_03581_gb300 as P  # noqa: E402
from oracle import oracle as O  # noqa: E402
from parity_util import first_mismatch, lockstep  # noqa: E402

ROWS_BYTES = 24 << 10       # 64 rows up to 128 topics, 8 at 1,000, 5 at 1,100, 2 at 3,000


def corpus(rng, lengths, V, a=1.0):
    off = np.zeros(len(lengths) + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    p = (1.0 + np.arange(V)) ** -a
    return rng.choice(V, size=int(off[-1]), p=p / p.sum()).astype(np.int32), off


def noalloc(s, w, off, sweeps, seed):
    import torch
    z = torch.empty(len(w), dtype=torch.int16, device="cuda")
    P.pulda_infer_noalloc(s.h, torch.from_numpy(w).cuda(), torch.from_numpy(off).cuda(), sweeps, seed, z)
    return z.cpu().numpy()


def main():
    assert os.path.realpath(P.LIB_PATH) == os.path.realpath(os.environ["PULDA_LIB"]), P.LIB_PATH
    # one document per warp, and per CTA; columns of some tens to several
    # hundred topics; counts past one plane; lengths around the groups and blocks
    for K, V in [(100, 200), (300, 120), (600, 60), (1000, 40), (1024, 300), (1100, 60), (3000, 40), (9000, 24)]:
        for coop in (-1, 1):
            rng = np.random.default_rng(K + V)
            lengths = [0, 1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 63, 65, 96, 97, 254, 257, 1500, 2600]
            lengths += list(rng.integers(100, 400, size=20 if K > 2000 else 60))
            w, off = corpus(rng, lengths, V, 0.7)
            w[off[18]:off[19]:2] = rng.integers(V // 2, V // 2 + 3, size=(off[19] - off[18] + 1) // 2)
            alpha = rng.uniform(0.05, 0.5, K).astype(np.float32)
            alpha[:2] = 8.0
            s, ch = lockstep(w, off, K, V, alpha, 0.02, seed=K, sweeps=2, check_counts_every=2, coop_min_len=coop)
            nnz = np.diff(s.word_tables()["col_ptr"])
            assert nnz[V // 2:].max() > 33 and nnz.max() > min(256, K // 2), nnz
            a, b = off[14], off[19]
            new, noff = np.ascontiguousarray(w[a:b]), off[14:20] - a
            zo = O.infer(ch.tables, new, noff, 2, 7)
            assert not first_mismatch(s.infer(new, noff, 2, seed=7), zo, noff)
            assert not first_mismatch(noalloc(s, new, noff, 2, 7), zo, noff)
            srv = P.Server(s, token_budget=20000, max_slots=16, slice_tokens=0)
            docs = {i: np.ascontiguousarray(w[off[i]:off[i + 1]]) for i in range(10, 20)}
            for i, words in docs.items():
                srv.submit(i, i, words, 2)
            got = {}
            while len(got) < len(docs):
                for r in srv.poll(timeout_ms=500):
                    assert r["status"] == 0
                    got[r["req_id"]] = r["z"]
            srv.close()
            for i, words in docs.items():
                assert np.array_equal(got[i], O.infer(ch.tables, words, np.array([0, len(words)]), 2, i)), (K, coop, i)
            s.close()
    # two documents per warp, columns of up to K topics
    for K in (100, 500, 1000):
        rng = np.random.default_rng(K)
        lengths = rng.integers(0, 24, size=90001)
        lengths[:6] = [15, 16, 17, 255, 400, 2600]
        w, off = corpus(rng, lengths, 100, 0.5)
        s, _ = lockstep(w, off, K, 100, 0.1, 0.01, seed=K, sweeps=1, check_tables=False, coop_min_len=-1)
        assert s.z_layout()["docs_per_warp"] == 2
        assert (np.diff(s.word_tables()["col_ptr"])[64:] > min(256, K // 2)).any()
        s.close()
    # batched chains of every form
    rng = np.random.default_rng(4)
    chains = []
    for i, K in enumerate([50, 200, 400, 900, 2000]):
        w, off = corpus(rng, np.append(rng.integers(20, 200, size=120), [700, 900]), 60, 0.7)
        chains.append(dict(w=w, doc_off=off, K=K, V=60, alpha=0.1, beta=0.01, seed=20 + i))
    for coop in (-1, 150):
        b = P.Batch(chains, coop_min_len=coop)
        b.sweep(3)
        for i, c in enumerate(chains):
            one = P.Sampler(c["w"], c["doc_off"], c["K"], c["V"], 0.1, 0.01, c["seed"], coop_min_len=coop).sweep(3)
            assert np.array_equal(b.z(i), one.z()), (coop, i)
            one.close()
        b.close()
    print("few rows: all cases passed")


if __name__ == "__main__":
    main()
