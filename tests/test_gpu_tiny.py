"""The single-launch kernel for n <= 64 at the edges of its widths (8, 16, 24, 32, 48, 64) and of its one
and four warps per block (608 restarts): trajectories within the FP32 tolerance 1e-5 of the oracle, exact
objectives and records, and the same bits when a run is split into calls."""
import numpy as np
import pytest

import oracle as O
import workloads as W
from paper_2509_21064_gb300 import sbo as S
from paper_2509_21064_gb300.build import build as build_lib
from _helpers import normwise, oracle_trajectory, to_gda_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build_lib()
    S.lib()


@pytest.mark.parametrize("n,B", [(1, 3), (8, 1), (9, 5), (16, 608), (17, 609), (24, 2), (25, 7), (32, 33), (33, 700), (48, 4),
                                 (49, 3), (64, 610)])
def test_tiny_widths(n, B):
    Q, c = W.dense_qubo(n, seed=n)
    p = W.dense_params(Q, restarts=B, iters=45, eval_every=10, seed=n)
    prm = to_gda_params(p)
    with S.Problem.dense(Q, c, precision=S.SBO_FP32) as P:
        P.start(prm)
        states = []
        for k in (1, 19, 10, 10, 5, 5):      # past T = 45: evaluations at 10, .., 40, 45, 50
            P.run(k)
            states.append(P.state())
        assert P.info()["kernel"] == S.KERNEL_TINY
        trace, (x, F, t, r), (Fr, tr) = P.trace(), P.best(), P.restart_best()
        ox, oy, _ = oracle_trajectory(Q, c, p, 45)
        for done, (X, Y) in zip((1, 20, 30, 40, 45), states):
            assert normwise(X, ox[done]).max() <= 1e-5 and normwise(Y, oy[done]).max() <= 1e-5
        F40 = O.objective_batch(Q, c, O.round_bits(states[3][0]))
        assert len(trace) == 6 and int(F40.min()) == int(trace[3])
        assert np.all(Fr <= F40) and int(Fr.min()) == F == int(trace.min()) == O.objective(Q, c, x)
        assert set(tr.tolist()) <= {10, 20, 30, 40, 45, 50}
        P.start(prm)
        P.run(50)
        X, Y = P.state()
        assert np.array_equal(X, states[-1][0]) and np.array_equal(Y, states[-1][1])
        assert np.array_equal(P.trace(), trace) and np.array_equal(P.restart_best()[0], Fr)
