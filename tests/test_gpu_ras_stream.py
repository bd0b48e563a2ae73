"""The RAS application's factor streams at the sizes where their layout
changes: one-row subdomains, levels of more than 32 rows, rows of more than
six entries per triangle (a 27-point stencil, a well with many perforations:
such rows take part in several groups), overlap 2, and a pattern that is not
symmetric (no row may then be left out of the sweeps).

The systems are diagonally dominant: the off-diagonal blocks of a row sum to
at most half its diagonal block in norm, so the triangular solves amplify a
relative rounding error of the factors by at most a few.  Bars, relative to
the largest output: 1e-10 in FP64, 1e-4 in FP32 (2^-24 times the sums'
lengths and the amplification leaves two orders of margin), 2^-6 with BF16
factor values (2^-9 each, times a bound of 8)."""
import numpy as np
import pytest

import oracle
import paper_1701_06254_gb300 as R

pytestmark = pytest.mark.gpu

BAR = {R.PREC_FP64: 1e-10, R.PREC_MIXED: 1e-4, R.PREC_MIXED_BF16: 2.0 ** -6}


def _system(nx, ny, nz, wide, wells, seed):
    """(rp, ci, val, b, key, first perforations): cells coupled to their 6 or
    26 neighbours, wells[k] = (i, j) perforating a whole column."""
    rng = np.random.default_rng(seed)
    n, nw = nx * ny * nz, len(wells)
    rows = [set() for _ in range(n + nw)]
    for c in range(n):
        i, j, k = c % nx, (c // nx) % ny, c // (nx * ny)
        for dk in (-1, 0, 1):
            for dj in (-1, 0, 1):
                for di in (-1, 0, 1):
                    if not wide and abs(di) + abs(dj) + abs(dk) > 1:
                        continue
                    a, b_, d = i + di, j + dj, k + dk
                    if 0 <= a < nx and 0 <= b_ < ny and 0 <= d < nz:
                        rows[c].add(a + nx * (b_ + ny * d))
    wc0 = []
    for w, (i, j) in enumerate(wells):
        rows[n + w].add(n + w)
        wc0.append(i + nx * j)
        for k in range(nz):
            c = i + nx * (j + ny * k)
            rows[n + w].add(c)
            rows[c].add(n + w)
    rp = np.zeros(n + nw + 1, np.int32)
    ci, val = [], []
    for r, cols in enumerate(rows):
        cols = sorted(cols)
        rp[r + 1] = rp[r] + len(cols)
        for c in cols:
            m = rng.uniform(-1.0, 1.0, (2, 2))
            if c == r:
                m = np.array([[1.0, 0.1], [-0.1, 1.0]]) + 0.05 * m
            else:
                m *= 0.2 / max(len(cols) - 1, 1)
            ci.append(c)
            val.append(m.reshape(-1))
    return (rp, np.array(ci, np.int32), np.concatenate(val), rng.standard_normal(2 * (n + nw)),
            rng.permutation(n).astype(np.float64), wc0)


@pytest.mark.parametrize("prec", [R.PREC_FP64, R.PREC_MIXED, R.PREC_MIXED_BF16], ids=["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("grid,wide,wells,opts", [
    ((1, 1, 1), False, [], {}),
    ((5, 1, 1), False, [], dict(tile_x=1, tile_y=1)),
    ((9, 6, 3), True, [(8, 5)], {}),
    ((8, 5, 40), False, [(1, 1), (6, 3)], {}),
    ((13, 11, 4), False, [(0, 0)], dict(overlap=2, tile_x=5, tile_y=3)),
    ((24, 18, 2), False, [], dict(tile_x=24, tile_y=18, reorder=0)),
], ids=["one_row", "line", "wide_stencil", "long_wells", "overlap2", "one_subdomain"])
def test_ras_matches_oracle(grid, wide, wells, opts, prec):
    rp, ci, val, b, key, wc0 = _system(*grid, wide, wells, seed=5)
    opts = dict(opts, decoupling=R.DEC_NONE, amg_coarse_max=2048)
    o = oracle.LinearSystem(*grid, len(wells), rp, ci, wc0, **opts)
    g = R.LinearSystem(*grid, len(wells), rp, ci, wc0, precision=prec, **opts)
    o.set(val, b, key); g.set(val, b, key)
    o.setup(); g.setup()
    x = np.random.default_rng(6).standard_normal(len(b))
    yo, yg = o.ras(x), g.apply(R.OP_RAS, x)
    assert np.abs(yg - yo).max() <= BAR[prec] * np.abs(yo).max()


def test_ras_keeps_every_row_of_an_unsymmetric_pattern():
    """Two wells coupled one way only (A_pp stays symmetric, which the AMG
    setup insists on): the second well's row reads the first's, not the
    other way round."""
    nx, ny, nz = 6, 4, 3
    wells = [(1, 1), (2, 1)]
    rp, ci, val, b, key, wc0 = _system(nx, ny, nz, False, wells, seed=9)
    n = nx * ny * nz
    q = int(rp[n + 2]) - 1                     # the second well's diagonal, its row's last entry
    ci = np.insert(ci, q, n).astype(np.int32)  # column of the first well before it
    val = np.insert(val, 4 * q, [0.1, 0.0, 0.0, 0.1])
    rp = rp.copy(); rp[n + 2] += 1
    opts = dict(decoupling=R.DEC_NONE, amg_coarse_max=2048)
    o = oracle.LinearSystem(nx, ny, nz, 2, rp, ci, wc0, **opts)
    g = R.LinearSystem(nx, ny, nz, 2, rp, ci, wc0, precision=R.PREC_FP64, **opts)
    o.set(val, b, key); g.set(val, b, key)
    o.setup(); g.setup()
    x = np.random.default_rng(7).standard_normal(len(b))
    yo, yg = o.ras(x), g.apply(R.OP_RAS, x)
    assert np.abs(yg - yo).max() <= 1e-10 * np.abs(yo).max()
