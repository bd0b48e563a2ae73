"""Large RAS subdomains: whole models as one subdomain, up to and beyond the
9,900 to 11,400 rows at which the tables that the factor streams are packed
with stop fitting in shared memory (then they lie in global memory).  Beyond
as before the streamed application and the recorded Arnoldi step are used,
and the application matches the oracle with the bars of test_gpu_ras_stream.
"""
import numpy as np
import pytest

import oracle
import paper_1701_06254_gb300 as R
import test_gpu_ras_stream

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [R.PREC_FP64, R.PREC_MIXED, R.PREC_MIXED_BF16], ids=["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("grid", [(1, 1, 11372), (1, 1, 11373), (4, 4, 700), (1, 1, 12700)],
                         ids=["column_below", "column_beyond", "tile_beyond", "column_12700"])
def test_large_subdomains_match_oracle(grid, prec):
    rp, ci, val, b, key, wc0 = test_gpu_ras_stream._system(*grid, False, [], seed=11)
    opts = dict(decoupling=R.DEC_NONE)
    o = oracle.LinearSystem(*grid, 0, rp, ci, wc0, **opts)
    g = R.LinearSystem(*grid, 0, rp, ci, wc0, precision=prec, **opts)
    o.set(val, b, key); g.set(val, b, key)
    o.setup(); g.setup()
    assert g.ras_count() == 1
    x = np.random.default_rng(12).standard_normal(len(b))
    yo, yg = o.ras(x), g.apply(R.OP_RAS, x)
    assert np.abs(yg - yo).max() <= test_gpu_ras_stream.BAR[prec] * np.abs(yo).max()
    y, its, rel = g.solve(1e-6)
    assert rel <= 1e-6 and g.graph_mode() == 1
