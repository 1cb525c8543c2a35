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


@pytest.mark.parametrize("repeat", [1, 3])
@pytest.mark.parametrize("scale", [1.0, 1e-25, 1e160, 1e-170, "special"])
@pytest.mark.parametrize("pk", [dict(epi_px=4.0, bits_per_table=3, n_tables=2), dict(epi_px=0.0, bits_per_table=0, n_tables=1),
                                dict(epi_px=300.0, bits_per_table=5, tau=60, top_k=16)])
def test_join_band_block_edges(ch, orc, pk, scale, repeat):  # noqa: F811
    """The band form of the join: blocks of 1 to 300 queries and candidates, by one CTA and by clusters; lines that
    are ordinary, tiny, overflow FP32 or FP64 once squared, and ones with key-points and matrices that are huge,
    infinite or NaN, where every decision is the FP64 expression's."""
    s = synth.random_set(516, SIZES[1:])
    n = len(SIZES) - 1
    pairs = np.array([(i, k) for i in range(n) for k in range(n)] * repeat, np.uint32)
    rng = np.random.default_rng(516)
    s.kpts = (rng.random((s.desc.shape[0], 2)) * [1920.0, 1080.0]).astype(np.float32)
    s.kpts[::7] = np.round(s.kpts[::7] / 64) * 64
    s.F = rng.standard_normal((len(pairs), 9)) * [1e-6, 1e-6, 1e-3, 1e-6, 1e-6, 1e-3, 1e-3, 1e-3, 1.0]
    s.F[::5] = [0, 0, 0, 0, 0, -1, 0, 1, 0]  # rows of equal y: candidates exactly on a line
    if scale == "special":
        v = np.float32([np.inf, -np.inf, np.nan, 1e20, -1e30, 3e38, 1e-42])
        s.kpts[3::11, 0] = rng.choice(v, s.kpts[3::11].shape[0])
        s.kpts[5::13, 1] = rng.choice(v, s.kpts[5::13].shape[0])
        s.F[1::4, 4] = rng.choice([np.inf, np.nan, 1e308, 1e-310], s.F[1::4].shape[0])
        s.F[2::4, :6] *= 1e-44
    else:
        s.F *= scale
    ctx, ds, off, got, _ = gpu_run(ch, s, pairs, tuning=(ch.CASHASH_KERNEL_JOIN, 4, 0), schedule=1, **pk)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    eoff, emt = orc.match_pairs(s.desc, s.img_off, codes, buckets, pairs, po, F=s.F, kpts=s.kpts)
    assert np.array_equal(off, eoff)
    assert np.array_equal(got, emt)
    ctx.close()
