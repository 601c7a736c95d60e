"""The dense-row z-step at the edges of its forms, against the oracle: every
topic, count and counter equal."""
import numpy as np
import pytest

from oracle import oracle as O
from parity_util import compare_tables, first_mismatch, lockstep

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
    p = (1.0 + np.arange(V)) ** -1.0
    return rng.choice(V, size=int(off[-1]), p=p / p.sum()).astype(np.int32), off


@pytest.mark.parametrize("coop", [-1, 1])
@pytest.mark.parametrize("K", [3, 4, 5, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1536, 1537, 4097])
def test_forms_and_record_rings(K, coop):
    """K around the words per lane (1, 2, 4, 8) and the chunks above 1024;
    lengths around the staged blocks (32), the record ring (96), one count
    plane (255) and the groups of rows; one document per warp and per CTA."""
    rng = np.random.default_rng(900 + K)
    lengths = [0, 1, 2, 3, 4, 5, 7, 8, 9, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 191, 192, 193, 254, 255, 256, 257, 1500]
    w, off = corpus(rng, lengths, 400)
    s, _ = lockstep(w, off, K, 400, rng.uniform(0.05, 0.5, K).astype(np.float32), 0.02, seed=K, sweeps=3, check_counts_every=3,
                    coop_min_len=coop)
    s.close()


@pytest.mark.parametrize("coop", [-1, 1])
@pytest.mark.parametrize("K", [2, 20, 600, 1100])
def test_counts_across_a_plane(K, coop):
    """Few topics carry most of long documents, so that counts pass 255 and
    come back within a pass, and lane sums pass 2^32."""
    rng = np.random.default_rng(K)
    lengths = [230, 258, 300, 520, 700, 5000]
    off = np.zeros(len(lengths) + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    w = rng.integers(0, 6, size=int(off[-1])).astype(np.int32)
    alpha = np.full(K, 0.01, np.float32)
    alpha[:2] = 20.0
    s, _ = lockstep(w, off, K, 40, alpha, 0.01, seed=5, sweeps=4, check_counts_every=4, coop_min_len=coop)
    s.close()


@pytest.mark.parametrize("K", [40, 1100])
def test_three_count_planes_beside_long_documents(K):
    """A document of 2^16 tokens or more (three planes, one warp) beside
    documents on CTAs."""
    rng = np.random.default_rng(11)
    w, off = corpus(rng, [70000, 3000, 65535, 100, 65536], 300)
    s, _ = lockstep(w, off, K, 300, 0.1, 0.01, seed=2, sweeps=1, check_tables=False, coop_min_len=0)
    s.close()


@pytest.mark.parametrize("coop", [-1, 1])
def test_weight_of_twenty_five_bits(coop):
    """phi so near 1 that its weight rounds to 2^24, which three bytes do not
    hold: the word is summed over its column."""
    import paper_1704_03581_gb300 as P
    n = (1 << 25) + 60000               # the row's draws sum to at least 2^25 (ten standard deviations)
    w = np.zeros(n, np.int32)
    w[5] = 1
    off = np.append(np.arange(0, n, 1 << 22), n).astype(np.int64)
    for seed in range(30):              # the other word drawn once: probability 0.37
        s = P.Sampler(w, off, 1, 2, 0.1, 0.01, seed=seed, coop_min_len=coop)
        s.phi_step()
        tables = s.word_tables()
        if tables["q"].max() == 1 << 24:
            break
        s.close()
    ch = O.Chain(w, off, 1, 2, 0.1, 0.01, seed=seed)
    ch.sweep_index += 1
    ch.phi_step(ch.sweep_index)
    assert tables["q"].max() == 1 << 24
    compare_tables(tables, ch)
    nw = np.array([0] * 40 + [1] + [0] * 300, np.int32)
    noff = np.array([0, 1, 41, len(nw)], np.int64)
    zg = s.infer(nw, noff, 1, seed=9)
    zo, stats = O.z_step(noff, nw, np.zeros(len(nw), np.int16), ch.tables, 9, 1)
    assert not first_mismatch(zg, zo, noff)
    st = s.stats()
    assert [st[k] for k in ("tokens", "a_branch", "sum_min", "zero_mass", "sum_inter", "docside")] == list(stats[:6])
    s.close()


def test_noalloc_schedules_every_length_class():
    """More documents than the GPU holds CTAs, of every length class, in
    arrival order: pulda_infer's topics."""
    import torch
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(3)
    w, off = corpus(rng, rng.integers(0, 60, size=300), 500)
    s = P.Sampler(w, off, 100, 500, 0.1, 0.01, seed=1)
    s.sweep(2)
    lengths = rng.integers(0, 40, size=20000)
    lengths[[7, 900, 19999]] = [66000, 700, 5000]
    nw, noff = corpus(rng, lengths, 500)
    z = torch.empty(len(nw), dtype=torch.int16, device="cuda")
    P.pulda_infer_noalloc(s.h, torch.from_numpy(nw).cuda(), torch.from_numpy(noff).cuda(), 2, 77, z)
    assert np.array_equal(z.cpu().numpy(), s.infer(nw, noff, 2, seed=77))
    s.close()


@pytest.mark.parametrize("K", [3, 128, 129, 257, 512, 513, 1000, 1024])
def test_two_documents_per_warp(K):
    """A pass over enough documents to go two per warp: uneven neighbours, empty
    documents, lengths around the 16-token blocks, counts past one plane."""
    rng = np.random.default_rng(K)
    lengths = rng.integers(0, 24, size=90001)
    lengths[:9] = [15, 16, 17, 31, 33, 255, 400, 2600, 2601]
    w, off = corpus(rng, lengths, 700)
    heavy = slice(int(off[7]), int(off[9]))
    w[heavy] = rng.integers(0, 4, size=heavy.stop - heavy.start)
    alpha = np.full(K, 0.05, np.float32)
    alpha[0] = 5.0
    s, _ = lockstep(w, off, K, 700, alpha, 0.01, seed=K, sweeps=2, check_tables=False, coop_min_len=-1)
    assert s.z_layout()["docs_per_warp"] == 2
    s.close()
