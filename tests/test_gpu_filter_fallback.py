"""GPU tests (-m gpu): fp64 in blocks of 64 where 16-bit bounds cannot filter the
relaxations (a vertex far from all others in every block, a large finite weight
for a missing edge, negative edges): bit for bit the phased driver's results,
which relax every step of every entry in order, and not slower than it."""
from __future__ import annotations

import numpy as np
import pytest

from fwtest import fw, gpu_solve

pytestmark = pytest.mark.gpu

PERSISTENT, PHASED = 1, 2


def _weights(n, kind, seed):
    r = np.random.RandomState(seed)
    W = 1 - r.random_sample((n, n))
    W[r.random_sample((n, n)) >= 0.5] = np.inf
    if kind == "far":
        W[17::64, :] = W[:, 17::64] = 1e9
    elif kind == "half":
        W[::2, :] *= 1e9
        W[:, ::2] *= 1e9
    elif kind == "no_edge":
        W = np.where(r.random_sample((n, n)) < 8.0 / n, 1 - r.random_sample((n, n)), 1e9)
    elif kind == "negative":  # by potentials: negative edges, no negative cycle
        pot = np.floor(4 * r.random_sample(n))
        W = np.floor(1 + 8 * r.random_sample((n, n))) + pot[:, None] - pot[None, :]
    np.fill_diagonal(W, 0)
    return W


# one CTA per SM up to 27 x 27 tiles (five per SM and round), two above
@pytest.mark.parametrize("n", [64, 191, 700, 27 * 64, 27 * 64 + 1])
@pytest.mark.parametrize("kind", ["uniform", "far", "half", "no_edge", "negative"])
def test_unfiltered_tiles_bit_for_bit(n, kind):
    import torch
    m = fw()
    W = _weights(n, kind, n)
    D, P = gpu_solve(W, bs=64, driver=PERSISTENT, extra_ld=4)
    Dr, Pr = gpu_solve(W, bs=64, driver=PHASED)
    assert D.tobytes() == Dr.tobytes() and np.array_equal(P, Pr)
    Dd, none = m.solve(torch.from_numpy(W).cuda(), m.Options.default(bs=64, driver=PERSISTENT),
                       with_pred=False)
    assert none is None and Dd.cpu().numpy().tobytes() == Dr.tobytes()


def _best_ms(W, driver):
    import torch
    m = fw()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    opt = m.Options.default(bs=64, driver=driver)
    best = 1e9
    for _ in range(4):
        ev[0].record()
        m.solve(W, opt)
        ev[1].record()
        ev[1].synchronize()
        best = min(best, ev[0].elapsed_time(ev[1]))
    return best


@pytest.mark.parametrize("n", [700, 2048])
@pytest.mark.parametrize("kind", ["far", "no_edge"])
def test_useless_bounds_cost_no_more_than_none(n, kind):
    """The phased driver relaxes the same tiles exactly, with three launches a
    round and nothing overlapped: the filter, where it is of no use, must not
    make the persistent driver slower than that (it was two to three times)."""
    import torch
    W = torch.from_numpy(_weights(n, kind, 3)).cuda()
    assert _best_ms(W, PERSISTENT) < 1.2 * _best_ms(W, PHASED)
