"""The bucket join with every number of CTAs that may share a pair (8, 4, 2 or
1, by the number of pairs and the SMs of the device), with and without the
band, against the oracle (match lists entry for entry: every result is an
integer, so the tolerance is zero)."""
import numpy as np
import pytest
import torch

import synth
from test_gpu_parity import ch, gpu_run, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu

# tiles of 32 queries that end inside, at and behind a CTA's share; fewer tiles than CTAs; empty images
SIZES = [300, 0, 1, 33, 256, 257, 65, 31, 96]


@pytest.mark.parametrize("pk", [dict(top_k=10), dict(bits_per_table=3, n_tables=2, top_k=2), dict(bits_per_table=5, top_k=16, tau=60),
                                dict(bits_per_table=0, n_tables=1, top_k=10), dict(epi_px=40.0, bits_per_table=3, n_tables=2),
                                dict(epi_px=300.0, bits_per_table=6, top_k=16)])
@pytest.mark.parametrize("ctas", [8, 4, 2, 1])
def test_join_cluster_sizes(ch, orc, pk, ctas):  # noqa: F811
    """The most pairs that clusters of `ctas` still take (two CTAs are resident per SM); one more than pairs of CTAs take."""
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    P = 2 * nsm // ctas if ctas > 1 else nsm + 1
    s = synth.random_set(1414, SIZES)
    n = len(SIZES)
    pairs = np.resize(np.array([(i, k) for i in range(n) for k in range(n)], np.uint32), (P, 2))
    if "epi_px" in pk:
        rng = np.random.default_rng(1414)
        s.kpts = (rng.random((s.desc.shape[0], 2)) * [1920.0, 1080.0]).astype(np.float32)
        s.F = rng.standard_normal((P, 9)) * [1e-6, 1e-6, 1e-3, 1e-6, 1e-6, 1e-3, 1e-3, 1e-3, 1.0]
    ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(ch.CASHASH_KERNEL_JOIN, 4, 0), schedule=1, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po, F=s.F, kpts=s.kpts)
    assert np.array_equal(off, eoff)
    assert np.array_equal(got, emt)
    ctx.close()
