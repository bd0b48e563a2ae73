"""Sizes at which the solver changes kernels, against the oracle with the bars
of the tests whose checks are used here: one-block scans end at 24,576 rows,
RAS takes two lanes per row in FP32 and BF16 up to 1,216 subdomains, and
BiCGSTAB's sums take a second block from 4,097 values on.
"""
import numpy as np
import pytest

import paper_1701_06254_gb300 as R
from paper_1701_06254_gb300 import inputs as I
import test_gpu_parity
import test_gpu_ras_stream
import test_gpu_solvers

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(48, 32, 16), (49, 32, 16)], ids=["24576", "25088"])
def test_setup_about_the_one_block_scan(shape):
    test_gpu_parity.test_setup_integer_work_is_bit_exact(lambda: I.case2(nx=shape[0], ny=shape[1], nz=shape[2]), dict())


@pytest.mark.parametrize("prec", [R.PREC_MIXED, R.PREC_MIXED_BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("grid", [(32, 38, 2), (35, 35, 2)], ids=["1216", "1225"])
def test_ras_about_one_wave_of_two_lanes(grid, prec):
    test_gpu_ras_stream.test_ras_matches_oracle(grid, False, [(3, 4)], dict(tile_x=1, tile_y=1), prec)


@pytest.mark.parametrize("prec", [R.PREC_FP64, R.PREC_MIXED_BF16], ids=["fp64", "bf16"])
@pytest.mark.parametrize("shape", [(16, 16, 8), (33, 31, 9)])
def test_bicgstab_of_several_blocks(shape, prec):
    """Solution and true residual; in BF16 the iteration count is the
    preconditioner's (25 to the oracle's 16 on the first grid at 1e-10)."""
    o, gl = test_gpu_solvers._shared(I.small_case(*shape, seed=23), 310, krylov=R.KRYLOV_BICGSTAB, precision=prec)
    o.ls.setup(); gl.setup()
    rco, yo, _, _ = o.ls.solve(1e-10)
    yg, _, relg = gl.solve(1e-10)
    assert rco == 0 and relg <= 1e-10
    _, _, _, db, _ = o.ls.get()
    assert np.linalg.norm(db - o.ls.mv(yg)) <= 1.0001e-10 * np.linalg.norm(db)
    assert np.abs(yg - yo).max() <= 1e-7 * np.abs(yo).max()
