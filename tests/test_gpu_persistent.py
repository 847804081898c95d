"""The persistent sweeps of the block solves against launches per depth, each forced through
the autotuner's cache file (the tuner itself takes whichever is the faster, which on small
systems are the launches).  The file is read once per process, so every run is a child."""

import json
import os
import subprocess
import sys

import numpy as np
import pytest

import workloads as W
from gpu_helpers import relerr
from oracle.ddps_oracle import DDPSOracle

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CHILD = r"""
import sys, numpy as np
import workloads as W
from gpu_helpers import dev, host
from paper_1008_1700_gb300 import Solver, native as N
from test_gpu_persistent import problems
name, prec, out = sys.argv[1:]
p = getattr(N, "DDPS_" + prec)
probs = problems(name)
S = Solver.from_systems([(q.rowptr, q.colind, q.values, q.block_ptr) for q in probs],
                        factor_prec=p, spike_prec=p, ghat_prec=p, inner_prec=p, tol_out=1e-9)
S.factor(dev(S.values_host))
y = dev(np.random.default_rng(9).standard_normal(S.n))
g = [host(S.block_solve(y)).copy() for _ in range(3)]  # plain, captured, replayed
x, info = S.solve(dev(np.concatenate([q.f for q in probs])))
np.savez(out, g=np.stack(g), x=host(x), ok=info["status"] == "DDPS_OK",
         level=S.tuning()["persistent_from_level"])
"""


def problems(name):
    if name == "slabs":
        return [W.small_convdiff_3d(16, [5, 6, 5])]
    return [W.small_convdiff_2d(24, 8, seed=60 + k) for k in range(40)]


@pytest.mark.parametrize("prec,bound", [("FP64", 1e-12), ("FP32", 1e-5)])
@pytest.mark.parametrize("name", ["slabs", "batch"])
def test_persistent_sweeps_match_launches_per_depth(name, prec, bound, tmp_path):
    cache = tmp_path / "tune.json"
    env = dict(os.environ, DDPS_TUNE_CACHE=str(cache),
               PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))

    def run(choice):
        if choice is not None:
            c = json.loads(cache.read_text())
            keys = [k for k in c if "|persist|" in k]
            assert len(keys) == 1
            c[keys[0]] = choice
            cache.write_text(json.dumps(c))
        out = tmp_path / f"out{choice}.npz"
        subprocess.run([sys.executable, "-c", CHILD, name, prec, str(out)], check=True, env=env,
                       timeout=300)
        return np.load(out)
    run(None)  # the tuner writes the file
    per_depth, persistent = run(0), run(1)
    assert per_depth["level"] == -1 and persistent["level"] >= 0
    assert per_depth["ok"] and persistent["ok"]
    for r in (per_depth, persistent):
        assert np.array_equal(r["g"][0], r["g"][1]) and np.array_equal(r["g"][0], r["g"][2])
    assert relerr(persistent["g"][0], per_depth["g"][0]) <= bound
    assert relerr(persistent["x"], per_depth["x"]) <= 1e-6
    probs = problems(name)
    p = probs[0]
    o = DDPSOracle(p.n, p.rowptr, p.colind, p.values, p.block_ptr, spikes=False)
    y = np.random.default_rng(9).standard_normal(sum(q.n for q in probs))[:p.n]
    assert relerr(persistent["g"][0][:p.n], o.block_solve(y)) <= bound


FIRST = r"""
import sys, time, numpy as np, torch
import workloads as W
from gpu_helpers import dev
from paper_1008_1700_gb300 import Solver, native as N
opts = dict(factor_prec=N.DDPS_FP32, spike_prec=N.DDPS_BF16X3, ghat_prec=N.DDPS_FP16, inner_prec=N.DDPS_FP32)
def factor_ms(probs, times):
    S = Solver.from_systems([(q.rowptr, q.colind, q.values, q.block_ptr) for q in probs], **opts)
    v, out = dev(S.values_host), []
    for _ in range(times):
        torch.cuda.synchronize()
        t = time.perf_counter()
        S.factor(v)
        torch.cuda.synchronize()
        out.append(1e3 * (time.perf_counter() - t))
    return out
factor_ms([W.small_convdiff_2d(12, 2)], 2)  # context, kernels
first, _, third = factor_ms([W.small_convdiff_2d(60 + k % 60, 8) for k in range(200)], 3)
print(first, third)
"""


def test_first_factorisation_of_a_batch_does_not_try_every_shape():
    """The autotuner of a handle's first factorisation stays within a few factorisations of a
    batch, whose depths hold tens of thousands of small fronts (every shape at every depth
    took as long as twenty)."""
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))
    env.pop("DDPS_TUNE_CACHE", None)
    r = subprocess.run([sys.executable, "-c", FIRST], check=True, env=env, timeout=300,
                       capture_output=True, text=True)
    first, third = (float(v) for v in r.stdout.split())
    assert first <= 6.0 * third, (first, third)
