"""The one-warp z-step's columns above 1,024 topics, against the oracle: columns
around the limit (K / 10) and of more than four entries a lane, in passes over
few and over many documents."""
import numpy as np
import pytest

from oracle import oracle as O  # noqa: F401
from parity_util import lockstep

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("docs", [30, 700])
@pytest.mark.parametrize("K", [1025, 1537, 2049, 4097, 5000, 16384])
def test_columns_around_the_limit(K, docs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03581_gb300 import build
    build.build()
    rng = np.random.default_rng(K + docs)
    lengths = rng.integers(0, 60000 // docs, size=docs)
    lengths[:6] = [0, 1, 31, 33, 255, 2000]
    off = np.zeros(docs + 1, np.int64)
    np.cumsum(lengths, out=off[1:])
    p = (1.0 + np.arange(60)) ** -1.0
    w = rng.choice(60, size=int(off[-1]), p=p / p.sum()).astype(np.int32)
    w[off[5]:off[6]:2] = 3              # counts past one plane
    alpha = rng.uniform(0.01, 0.1, K).astype(np.float32)
    alpha[[0, K - 1]] = 60.0
    s, _ = lockstep(w, off, K, 60, alpha, 0.01, seed=K, sweeps=2, check_counts_every=2, coop_min_len=-1)
    n_w = np.diff(s.word_tables()["col_ptr"])
    assert n_w.max() > max(128, K // 10) and ((n_w > 128) & (n_w <= max(160, K // 10))).any(), n_w
    s.close()
