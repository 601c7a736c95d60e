"""Launch reports say what runs: the layout of a corpus of few documents, all on
CTAs, and the warps per CTA of the one-launch batched form."""
import numpy as np
import pytest

import bench

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


@pytest.mark.parametrize("docs,kw,one_warp", [(100, {}, 0), (100, dict(coop_min_len=-1), 100), (100, dict(docs_per_warp=4), 0),
                                              (5000, {}, 5000)])
def test_z_layout(docs, kw, one_warp):
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(docs)
    w, off = corpus(rng, rng.integers(1, 100, size=docs), 300)
    s = P.Sampler(w, off, 20, 300, 0.1, 0.01, seed=1, **kw)
    lay = s.z_layout()
    assert lay["one_warp_docs"] == one_warp, lay
    assert bench.every_document_on_a_cta(lay) == (docs == 100 and not kw)
    # one z-step launch in each: nothing is long enough for CTAs beside the others
    assert bench.kernels_per_sweep(w, 0, lay) == bench.kernels_per_sweep(w, 0)
    s.close()


def test_one_launch_form_reports_its_warps():
    """At K = 9,000 eight warps' counts pass 160 KB: the z-step runs four."""
    import paper_1704_03581_gb300 as P
    rng = np.random.default_rng(1)
    w, off = corpus(rng, rng.integers(1, 100, size=50), 100)
    b = P.Batch([dict(w=w, doc_off=off, K=9000, V=100, alpha=0.1, beta=0.01, seed=3)], coop_min_len=-1, batch_form=2)
    b.sweep(3)
    assert b.tuning()[0] == 4 and b.tuning()[3]
    one = P.Sampler(w, off, 9000, 100, 0.1, 0.01, seed=3).sweep(3)
    assert np.array_equal(b.z(0), one.z())
    one.close()
    b.close()
