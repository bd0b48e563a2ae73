"""A singular block in a subdomain: Inf and NaN stay in the rows that depend
on it.  Two layers without a connection between them, in one subdomain (and in
the same groups of the factor stream); the first cell's block of layer 0 is
singular, so the factors of layer 0 are not finite, while layer 1 is solved
as before: the application is finite where the oracle's is, with the bars of
test_gpu_ras_stream there.  The rows' order is random, so that a lane's row
often has fewer entries than the row of the other layer it had before.
"""
import numpy as np
import pytest

import oracle
import paper_1701_06254_gb300 as R
import test_gpu_ras_stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [R.PREC_FP64, R.PREC_MIXED, R.PREC_MIXED_BF16], ids=["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("wide", [False, True], ids=["7_point", "27_point"])
@pytest.mark.parametrize("nsub", [1, 1300], ids=["two_lanes", "one_lane"])
def test_singular_block_stays_in_its_rows(wide, nsub, prec):
    nx, ny = (13, 10) if nsub == 1 else (52, 100)
    lay = [test_gpu_ras_stream._system(nx, ny, 1, wide, [], seed=13 + k) for k in range(2)]
    n1 = nx * ny
    rp = np.concatenate([lay[0][0], lay[0][0][-1] + lay[1][0][1:]]).astype(np.int32)
    ci = np.concatenate([lay[0][1], n1 + lay[1][1]]).astype(np.int32)
    val = np.concatenate([lay[0][2], lay[1][2]])
    b = np.concatenate([lay[0][3], lay[1][3]])
    key = np.random.default_rng(15).permutation(2 * n1).astype(np.float64)
    key[0] = 2.0 * n1                                    # cell 0 first: its L columns are not finite either
    val[:4] = [1.0, 0.0, 0.0, 0.0]                       # cell 0's diagonal block, its row's first entry
    assert ci[0] == 0
    opts = dict(decoupling=R.DEC_NONE, reorder=1)
    opts.update(dict(tile_x=nx, tile_y=ny) if nsub == 1 else dict(tile_x=2, tile_y=2))
    o = oracle.LinearSystem(nx, ny, 2, 0, rp, ci, [], **opts)
    g = R.LinearSystem(nx, ny, 2, 0, rp, ci, [], precision=prec, **opts)
    o.set(val, b, key); g.set(val, b, key)
    o.setup(); g.setup()
    assert g.ras_count() == nsub
    x = np.random.default_rng(14).standard_normal(len(b))
    yo, yg = o.ras(x), g.apply(R.OP_RAS, x)
    ok = np.isfinite(yo)
    assert ok[2 * n1:].all() and not ok[:2 * n1].all()
    assert np.array_equal(np.isfinite(yg), ok)
    assert np.abs(yg - yo)[ok].max() <= test_gpu_ras_stream.BAR[prec] * np.abs(yo[ok]).max()
