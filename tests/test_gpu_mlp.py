"""The learned-guess network's CUDA kernels (forward, backward, Adam) against
the FP64 oracle network on the same parameters and data."""

import numpy as np
import pytest
import torch

from oracle import mlp_oracle as M
from paper_1008_1700_gb300 import native as N

pytestmark = pytest.mark.gpu


def _flat(params):
    return np.concatenate([np.concatenate([W.ravel(), b]) for W, b in params])


def _setup(seed, d_in=3, hidden=16, layers=3, d_out=20, B=6):
    rng = np.random.default_rng(seed)
    params = M.init_params(d_in, d_out, hidden=hidden, layers=layers, seed=seed)
    params = [(W + 0.05 * rng.standard_normal(W.shape), b + 0.1 * rng.standard_normal(b.shape))
              for W, b in params]
    X = rng.standard_normal((B, d_in))
    T = rng.standard_normal((B, d_out))
    return params, X, T, (d_in, hidden, layers, d_out, B)


def _dev(a):
    return torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda").contiguous()


@pytest.mark.parametrize("seed", [0, 1, 2])
def test_forward_and_gradients_match_oracle(seed):
    params, X, T, (d_in, hidden, layers, d_out, B) = _setup(seed)
    p = _dev(_flat(params))
    assert p.numel() == N.ddps_mlp_param_count(d_in, hidden, layers, d_out)
    ws = torch.empty(N.ddps_mlp_workspace_bytes(d_in, hidden, layers, d_out, B), dtype=torch.uint8,
                     device="cuda")
    Y = torch.empty(B, d_out, dtype=torch.float32, device="cuda")
    N.ddps_mlp_forward(p, d_in, hidden, layers, d_out, _dev(X), B, Y, ws)
    Yo, _ = M.forward(params, X)
    assert np.max(np.abs(Y.cpu().numpy() - Yo)) <= 1e-5 * max(1.0, np.max(np.abs(Yo)))
    g = torch.zeros_like(p)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    N.ddps_mlp_backward(p, d_in, hidden, layers, d_out, _dev(X), _dev(T), B, g, loss, ws)
    go = _flat(M.backward(params, X, T))
    gg = g.cpu().numpy()
    assert np.linalg.norm(gg - go) <= 1e-5 * np.linalg.norm(go)
    assert abs(loss.item() - M.loss(params, X, T)) <= 1e-5 * M.loss(params, X, T)


def test_adam_matches_oracle():
    params, X, T, (d_in, hidden, layers, d_out, B) = _setup(5)
    p = _dev(_flat(params))
    state = {}
    m = torch.zeros_like(p)
    v = torch.zeros_like(p)
    for step in (1, 2, 3):
        grads = M.backward(params, X, T)
        g = _dev(_flat(grads))
        N.ddps_mlp_adam(p, g, m, v, p.numel(), 1e-2, 0.9, 0.999, 1e-8, step)
        M.adam_step(params, grads, state, lr=1e-2)
    assert np.max(np.abs(p.cpu().numpy() - _flat(params))) <= 1e-5


@pytest.mark.parametrize("d_in,hidden,layers,d_out,B", [
    (1, 256, 3, 129, 1),      # one vector: a warp per four rows, a ragged last group
    (2, 33, 2, 130, 4),       # rows that are not 16-byte aligned
    (2, 256, 3, 2500, 5),     # the smallest batch of the tiled products
    (3, 48, 1, 31, 64),       # one hidden layer, every product small
    (2, 256, 3, 5003, 100),   # wide output: K splits with a remainder, ragged tiles
    (2, 300, 2, 1024, 130),   # more than one K stage of the small product
])
def test_shapes_match_oracle(d_in, hidden, layers, d_out, B):
    """Forward and gradients at the edges of the kernels' tiles: sums of at most
    5,003 FP32 products, whose rounding stays below 1e-5 of the result's norm."""
    params, X, T, _ = _setup(3, d_in, hidden, layers, d_out, B)
    p = _dev(_flat(params))
    ws = torch.empty(N.ddps_mlp_workspace_bytes(d_in, hidden, layers, d_out, B), dtype=torch.uint8,
                     device="cuda")
    Y = torch.empty(B, d_out, dtype=torch.float32, device="cuda")
    N.ddps_mlp_forward(p, d_in, hidden, layers, d_out, _dev(X), B, Y, ws)
    Yo, _ = M.forward(params, X)
    assert np.linalg.norm(Y.cpu().numpy() - Yo) <= 1e-5 * np.linalg.norm(Yo)
    g = torch.full_like(p, float("nan"))
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    N.ddps_mlp_backward(p, d_in, hidden, layers, d_out, _dev(X), _dev(T), B, g, loss, ws)
    go = _flat(M.backward(params, X, T))
    assert np.linalg.norm(g.cpu().numpy() - go) <= 1e-5 * np.linalg.norm(go)
    assert abs(loss.item() - M.loss(params, X, T)) <= 1e-5 * M.loss(params, X, T)


@pytest.mark.parametrize("name,size", [("ordinary", 1.0), ("tiny", 1e-21), ("huge", 3e17), ("one_square_overflows", 0.0),
                                       ("mixed", -1.0)])
def test_loss_keeps_fp64_sums(name, size):
    """The loss of a network that answers 0 is the targets' mean square: the float nearest to
    it, for any size whose mean square is a float, also where single squares are not."""
    d_in, hidden, layers, d_out, B = 2, 16, 1, 300, 70
    rng = np.random.default_rng(4)
    T = rng.uniform(0.5, 1.0, (B, d_out)) * (size if size > 0 else 1.0)
    if name == "one_square_overflows":
        T[B // 2, d_out // 2] = 3e19
    if name == "mixed":
        T *= 10.0 ** rng.integers(-18, 3, T.shape)
    T = T.astype(np.float32)
    p = torch.zeros(N.ddps_mlp_param_count(d_in, hidden, layers, d_out), device="cuda")
    ws = torch.empty(N.ddps_mlp_workspace_bytes(d_in, hidden, layers, d_out, B), dtype=torch.uint8,
                     device="cuda")
    g, loss = torch.zeros_like(p), torch.zeros(1, device="cuda")
    N.ddps_mlp_backward(p, d_in, hidden, layers, d_out, _dev(rng.standard_normal((B, d_in))), _dev(T), B,
                        g, loss, ws)
    exact = 0.5 / B * np.sum(np.longdouble(T) ** 2)
    # the rounding to a float (or to a denormal one) and FP64 sums
    assert abs(float(loss.item()) - exact) <= (2.0 ** -24 + 1e-12) * exact + 2.0 ** -150 * 1.01
