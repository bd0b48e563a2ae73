"""One warm-start network used by several callers at a time: simulators in
threads of their own (their solves return before the network's work on the
shared activations is done) and a caller of the network itself.  Every result
must have the bits that it has with a network of its own, on grids of one
size (no buffer moves) and of two.
"""
import threading

import numpy as np
import pytest

import paper_1701_06254_gb300 as R
from paper_1701_06254_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _network():
    ws = R.WarmStart(seed=41)
    rng = np.random.default_rng(41)
    ws.set_params(ws.params() + 0.02 * rng.standard_normal(ws.params().size).astype(np.float32))
    return ws


def _states(case, ws, steps):
    g = R.Sim(case, precision=R.PREC_MIXED)
    g.init_hydrostatic()
    g.attach_warm_start(ws)
    out = []
    for _ in range(steps):
        g.advance(1)
        out.append(np.concatenate(g.get_state()[:3]))
    return out, g.stats()["linear_solves"]


@pytest.mark.parametrize("shapes", [[(12, 11, 5), (12, 11, 5)], [(12, 11, 5), (9, 14, 4)]], ids=["one_size", "two_sizes"])
def test_shared_network_gives_the_bits_of_a_network_each(shapes):
    cases = [I.small_case(*s, seed=60 + k) for k, s in enumerate(shapes)]
    steps = 6
    alone = [_states(c, _network(), steps) for c in cases]
    nx, ny, nz = shapes[0]
    F = np.random.default_rng(42).standard_normal((nz, ny, nx, 8)).astype(np.float32)
    ws = _network()
    y0 = ws.forward(F)
    got, ys, errors = [None] * len(cases), [], []
    running = threading.Event()
    running.set()

    def step(k):
        try:
            got[k] = _states(cases[k], ws, steps)
        except Exception as e:                     # reported by the main thread
            errors.append(e)

    def call():
        try:
            while running.is_set():
                ys.append(ws.forward(F))
        except Exception as e:
            errors.append(e)

    sims = [threading.Thread(target=step, args=(k,)) for k in range(len(cases))]
    caller = threading.Thread(target=call)
    for t in sims + [caller]:
        t.start()
    for t in sims:
        t.join()
    running.clear()
    caller.join()
    assert not errors, errors
    for (a, na), (b, nb) in zip(alone, got):
        assert na == nb > 0
        for x, y in zip(a, b):
            assert np.array_equal(x, y)
    assert ys and all(np.array_equal(y, y0) for y in ys)
