"""Several right-hand sides iterated together (one pass over G^ for up to four vectors)
against the same right-hand sides solved one at a time: the same iteration counts, solutions
within the outer tolerance, for one and for several systems in a handle, with a zero
right-hand side, an initial guess that is the answer, and group sizes 2, 3, 4 and 4 + rest."""

import numpy as np
import pytest

import workloads as W
from gpu_helpers import dev, host, make_solver
from paper_1008_1700_gb300 import Solver, native as N

pytestmark = pytest.mark.gpu

FORMS = {
    "fp16": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP16,
                 inner_prec=N.DDPS_FP32),
    "bf16_inner64": dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_FP32, ghat_prec=N.DDPS_BF16,
                         inner_prec=N.DDPS_FP64),
    "fp32_factors64": dict(factor_prec=N.DDPS_FP64, spike_prec=N.DDPS_FP64, ghat_prec=N.DDPS_FP32,
                           inner_prec=N.DDPS_FP32, use_graphs=0),
}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("nrhs", [2, 3, 4, 6])
@pytest.mark.parametrize("systems", [1, 2])
def test_together_equals_one_at_a_time(form, nrhs, systems):
    probs = [W.small_convdiff_3d(s, c) for s, c in ((27, [9, 8, 10]), (22, [7, 8, 7]))[:systems]]
    opts = dict(FORMS[form], tol_out=1e-11)
    if systems == 1:
        S = make_solver(probs[0], **opts)
    else:
        S = Solver.from_systems([(p.rowptr, p.colind, p.values, p.block_ptr) for p in probs], **opts)
        S.factor(dev(S.values_host))
    rng = np.random.default_rng([nrhs, systems])
    f = rng.uniform(-1.0, 1.0, (nrhs, S.n))
    f[1] = 0.0
    one = [S.solve(dev(v)) for v in f]
    assert all(i["status"] == "DDPS_OK" for _, i in one)
    x, info = S.solve(dev(f))
    assert info["status"] == "DDPS_OK"
    xs = np.stack([host(v) for v, _ in one])
    # both residuals are below 1e-11 |f|, the condition numbers below 27^2 / 2
    assert np.max(np.abs(host(x) - xs)) <= 2e-11 * 400 * np.max(np.abs(xs))
    assert np.all(host(x)[1] == 0.0)
    assert info["outer_iterations"] == max(i["outer_iterations"] for _, i in one)
    assert info["precond_applies"] == sum(i["precond_applies"] for _, i in one)
    assert abs(info["inner_iterations"] - sum(i["inner_iterations"] for _, i in one)) <= nrhs
    # initial guesses: the answers need no iteration
    y, again = S.solve(dev(f), x0=x)
    assert again["precond_applies"] == 0 and np.array_equal(host(y), host(x))
    S.close()


def test_workspace_is_for_the_right_hand_sides_asked_for():
    """Two right-hand sides take room for two; four, later, for four and no more; solutions
    and counts after the workspace has grown are those of a new handle."""
    P = W.small_convdiff_3d(27, [9, 8, 10])
    f = np.random.default_rng(4).uniform(-1.0, 1.0, (4, P.n))
    held = lambda S: N.ddps_get_sizes(S.h)["device_bytes"]
    S = make_solver(P, **FORMS["fp16"])
    b0 = held(S)
    x2, _ = S.solve(dev(f[:2]))
    b2 = held(S) - b0
    x4, i4 = S.solve(dev(f))
    b4 = held(S) - b0
    assert 0 < b2 <= 0.55 * b4
    again, _ = S.solve(dev(f[:2]))
    assert held(S) - b0 == b4 and np.array_equal(host(again), host(x2))
    T = make_solver(P, **FORMS["fp16"])
    c0 = held(T)
    y4, j4 = T.solve(dev(f))
    assert held(T) - c0 == b4 and np.array_equal(host(y4), host(x4))
    assert i4["inner_iterations"] == j4["inner_iterations"]
    S.close()
    T.close()
