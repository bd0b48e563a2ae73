"""How a BiCGSTAB solve ends other than by converging in one go: breakdown,
non-finite values, the iteration cap, restarts from the true residual, an
initial guess.  The decisions are taken from scalars that the device posts.
"""
import numpy as np
import pytest

import paper_1701_06254_gb300 as R
from paper_1701_06254_gb300 import inputs as I
from test_gpu_solvers import _shared

pytestmark = pytest.mark.gpu

BOTH = pytest.mark.parametrize("prec", [R.PREC_FP64, R.PREC_MIXED_BF16], ids=["fp64", "bf16"])


def _system(prec, scale=1.0, **opts):
    """A small shared system with its right-hand side scaled, without
    decoupling (which would scale the rows)."""
    opts = dict(opts, krylov=R.KRYLOV_BICGSTAB, precision=prec, decoupling=R.DEC_NONE)
    o, gl = _shared(I.small_case(11, 7, 4, seed=22), 340, **opts)
    rp, ci, val, b, key = o.system()
    gl.set(val, scale * b, key)
    gl.setup()
    return gl, scale * b


@pytest.mark.timeout(120)
def test_rhs_below_the_fp32_range():
    """2^-200 times a right-hand side.  FP64: every product and sum scales
    exactly, so does the solution.  Mixed precision: the preconditioner's
    input is zero in FP32, so the first iteration breaks down, and a restart
    would only repeat it: the solve ends with the zero vector it started from."""
    s = 2.0 ** -200
    y, its, rel = _system(R.PREC_FP64)[0].solve(1e-8)
    ys, its_s, rel_s = _system(R.PREC_FP64, s)[0].solve(1e-8)
    assert its_s == its > 0 and rel_s == rel <= 1e-8
    assert np.array_equal(ys, s * y)
    ym, its, rel = _system(R.PREC_MIXED_BF16, s)[0].solve(1e-8)
    assert its == 0 and rel == 1.0 and not ym.any()


def test_non_finite_values_are_errors():
    """NaN in the right-hand side; a right-hand side beyond the FP32 range
    in mixed precision (the first preconditioned vector is not finite)."""
    for prec, scale in ((R.PREC_FP64, np.nan), (R.PREC_MIXED_BF16, np.nan), (R.PREC_MIXED_BF16, 2.0 ** 200)):
        gl, _ = _system(prec, scale)
        with pytest.raises(R.SimError) as e:
            gl.solve(1e-8)
        assert e.value.code == 5          # SIM_ERR_NAN


@BOTH
def test_iteration_cap(prec):
    """At most max_lin iterations, and the residual that is reported is the
    solution's own."""
    gl, b = _system(prec, max_lin=2)
    y, its, rel = gl.solve(1e-12)
    assert its == 2 and rel > 1e-12
    assert rel == pytest.approx(gl.residual_norm(y) / np.linalg.norm(b), rel=1e-6)


@BOTH
def test_restart_from_the_true_residual(prec):
    """A tolerance below what FP64 rounding lets the true residual reach: the
    recursive residual meets it, the true one does not, and the solve goes on
    from the true residual until the cap."""
    gl, b = _system(prec, max_lin=200)
    y, its, rel = gl.solve(1e-18)
    assert its == 200 and 1e-18 < rel <= 1e-13      # about 1e3 roundings of 2^-53
    assert rel == pytest.approx(gl.residual_norm(y) / np.linalg.norm(b), rel=1e-6)


@BOTH
def test_initial_guess(prec):
    """Every solve from the previous step's first update (a fresh network
    predicts zero and leaves that guess): a whole run against the oracle's
    with the bars of the runs without a guess."""
    import oracle
    c = I.small_case(11, 7, 4, seed=22)
    o = oracle.Sim(c, krylov=R.KRYLOV_BICGSTAB)
    g = R.Sim(c, krylov=R.KRYLOV_BICGSTAB, precision=prec)
    o.init_hydrostatic(); g.init_hydrostatic()
    g.attach_warm_start(R.WarmStart(seed=2))
    for k in range(4):
        assert o.advance(1) == 0
        g.advance(1)
        po, so, _, to = o.get_state()
        pg, sg, _, tg = g.get_state()
        assert tg == to
        assert np.max(np.abs(pg - po) / np.abs(po)) <= 1e-6, k
        assert np.max(np.abs(sg - so)) <= 1e-6, k
    st = g.stats()
    assert st["ws_fallback"] == st["linear_solves"] > 0 and st["ws_r0"] < st["linear_solves"]
