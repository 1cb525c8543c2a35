"""The bucket join at the sizes where its blocks, clusters and lists have their
edges, against the oracle (match lists entry for entry: every result is an
integer, so the tolerance is zero)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu

# buckets of a few, half a warp's, a warp's and more queries; more candidates than are staged at a time
SIZES = [0, 1, 16, 17, 32, 33, 64, 65, 300]


@pytest.mark.parametrize("repeat", [1, 2, 4, 8])
@pytest.mark.parametrize("pk", [dict(bits_per_table=0, n_tables=1, top_k=10), dict(bits_per_table=3, n_tables=2, top_k=2),
                                dict(bits_per_table=5, n_tables=8, top_k=16, tau=60), dict(top_k=10, code_bits=64)])
def test_join_block_and_cluster_edges(ch, orc, pk, repeat):  # noqa: F811
    """Every ordered pair of the images, the list repeated so that a pair is shared by clusters of 2 to 8
    CTAs, or taken by one CTA; both the first launch (calibrated) and a second one (learned thresholds)."""
    s = synth.random_set(515, SIZES)
    n = len(SIZES)
    pairs = np.array([(i, k) for i in range(n) for k in range(n)][3:] * repeat, np.uint32)
    if repeat == 1:
        pairs = pairs[-30:]
    ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(ch.CASHASH_KERNEL_JOIN, 4, 0), schedule=1, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po)
    assert np.array_equal(off, eoff)
    assert np.array_equal(got, emt)
    ctx.close()
