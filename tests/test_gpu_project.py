"""The projection at the edges of its tiles and row halves, and on matrices whose
rows differ in scale, against the oracle (codes and buckets are bits: exact)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import ch, oparams, oracle_codes  # noqa: F401

pytestmark = pytest.mark.gpu


def _compare(ch, orc, s, pk):  # noqa: F811
    p = ch.cashash_default_params(**pk)
    ctx = ch.cashash_create(p, s.R)
    ds = ch.DeviceSet(p, s.img_off, s.desc, s.kpts)
    po = oparams(orc, pk)
    mu, codes, buckets = oracle_codes(orc, s.desc, s.R, po)
    for _ in range(3):
        ds.codes.zero_()
        ch.cashash_build_codes(ctx, ds)
        assert ch.cashash_sync_status(ctx) == ch.CASHASH_OK
        assert np.array_equal(ds.codes_np(), codes)
        assert np.array_equal(ds.buckets_np(po.n_tables), buckets)
    sq = (s.desc.astype(np.int64) ** 2).sum(axis=1)
    assert np.array_equal(ds.sqnorm.cpu().numpy().astype(np.int64), sq)
    rows = po.code_bits + po.n_tables * po.bits_per_table
    approx, bound = ch.cashash_projection_bounds(ctx, ds, 0, min(ds.n, 2000))
    v = orc.projections(s.desc[:2000], mu, s.R, rows)
    err = np.abs(approx.cpu().numpy().astype(np.float64) - v)
    ctx.close()
    return err, bound.cpu().numpy().astype(np.float64)


# 32, 95, 96, 97, 112, 176 and 192 rows of R
@pytest.mark.parametrize("pk", [dict(code_bits=32, n_tables=1, bits_per_table=0), dict(code_bits=64, n_tables=8, bits_per_table=4),
                                dict(code_bits=32, n_tables=7, bits_per_table=9 - 2), dict(code_bits=96, n_tables=1, bits_per_table=1),
                                dict(code_bits=64, n_tables=8, bits_per_table=6, precision=1), dict(precision=1),
                                dict(n_tables=8, bits_per_table=8)])
@pytest.mark.parametrize("n", [1, 127, 129, 20000])
def test_projection_tiles_and_rows(ch, orc, pk, n):  # noqa: F811
    err, bound = _compare(ch, orc, synth.random_set(717, [n]), pk)
    assert (err <= bound).all()


@pytest.mark.parametrize("precision", [0, 1])
def test_projection_scaled_rows(ch, orc, precision):  # noqa: F811
    """Rows of zeros, of one entry, of tiny, huge and mixed magnitudes, and constant descriptors."""
    s = synth.random_set(718, [700, 900])
    s.desc[:40] = 255
    s.desc[40:80] = 0
    R = np.array(s.R, np.float64)
    R[0] = 0.0
    R[1] = 0.0
    R[1, 77] = 3.0
    R[2] *= 1e-300
    R[3] *= 1e300
    R[4] *= 1e-38
    R[5] *= np.exp2(np.arange(128) - 64.0)
    R[6] = 512.0 * np.sign(R[6])
    R[7] = 511.99999999
    R[130] *= 2.0 ** 40
    R[131, 5] = 1e6
    R[132] = 5e-324
    s.R = R
    err, bound = _compare(ch, orc, s, dict(precision=precision))
    fin = [b for b in range(176) if b not in (2, 3, 132)]  # (1e-300 and 1e300 leave the range of the FP32 diagnostic)
    assert (err[:, fin] <= bound[:, fin]).all()
