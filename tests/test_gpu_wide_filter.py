"""GPU tests (-m gpu): the persistent driver's kernels of fp32 (steps in groups
of four), fp64 (blocks of 64 filtered by 16-bit bounds) and int64 give, bit for bit, the
distances and predecessors of the phased driver's kernels, which relax every
step of every entry in order: at tile edges, with ties, with missing edges, over
wide ranges of magnitude (bounds clamped, or zero), and distances alone."""
from __future__ import annotations

import numpy as np
import pytest

from fwtest import fw, gpu_solve

pytestmark = pytest.mark.gpu

PERSISTENT, PHASED = 1, 2


def _weights(dtype, n, kind, seed):
    r = np.random.RandomState(seed)
    integer = np.issubdtype(dtype, np.integer)
    u = r.random_sample((n, n))
    if kind == "uniform":
        W = 1 + u * (1e12 if integer else 1)
    elif kind == "ties":
        W = np.floor(1 + 4 * u)
    elif kind == "magnitudes":  # 12 (int64: 15) orders of magnitude
        W = np.exp(u * 34) if integer else np.exp((u - 0.5) * 28)
    elif kind == "tiny":  # below every bound's resolution beside some large edges
        W = np.where(r.random_sample((n, n)) < 0.5, 1 + 3 * u, 1e9 + 1e6 * u) * (1 if integer else 1e-6)
    else:
        W = 1 + 99 * u
    W = W.astype(dtype)
    inf = (1 << 61) if integer else np.inf
    p = 0.03 if kind == "sparse" else 0.7
    W[r.random_sample((n, n)) >= p] = inf
    np.fill_diagonal(W, 0)
    return W


@pytest.mark.parametrize("kind", ["uniform", "ties", "magnitudes", "tiny", "sparse"])
@pytest.mark.parametrize("dtype,bs", [(np.float32, 32), (np.float32, 64), (np.float32, 128),
                                      (np.float64, 32), (np.float64, 64), (np.int64, 32),
                                      (np.int64, 64)])
def test_drivers_agree_bit_for_bit(dtype, bs, kind):
    for n in (bs, 2 * bs + 1, 5 * bs - 3):
        W = _weights(dtype, n, kind, seed=n + bs)
        D, P = gpu_solve(W, bs=bs, driver=PERSISTENT, extra_ld=4)
        Dr, Pr = gpu_solve(W, bs=bs, driver=PHASED)
        assert D.tobytes() == Dr.tobytes() and np.array_equal(P, Pr)
        import torch
        m = fw()
        Dd, none = m.solve(torch.from_numpy(W).cuda(),
                           m.Options.default(bs=bs, driver=PERSISTENT), with_pred=False)
        assert none is None and Dd.cpu().numpy().tobytes() == Dr.tobytes()


@pytest.mark.parametrize("dtype", [np.float32, np.float64, np.int64])
def test_negative_cycle_across_tiles(dtype):
    """A negative cycle through vertices of different tiles is reported."""
    m = fw()
    W = _weights(dtype, 200, "sparse", seed=4)
    W[5, 70], W[70, 140], W[140, 5] = 1, 1, -10
    with pytest.raises(m.FWError) as e:
        gpu_solve(W, bs=64)
    assert e.value.code == 4
    gpu_solve(_weights(dtype, 90, "uniform", seed=5), bs=64)  # the status was cleared


@pytest.mark.parametrize("dtype", [np.int32, np.float32])
@pytest.mark.parametrize("n", [64 * 42, 64 * 42 + 1, 64 * 44 - 3])
def test_two_ctas_per_sm(dtype, n):
    """Blocks of 64 with 32-bit elements, around the size from which two CTAs
    share an SM."""
    W = _weights(np.float32, n, "small", seed=n)
    if dtype is np.int32:
        W = np.where(np.isinf(W), 1 << 29, W).astype(np.int32)
    D, P = gpu_solve(W, bs=64, driver=PERSISTENT)
    Dr, Pr = gpu_solve(W, bs=64, driver=PHASED)
    assert D.tobytes() == Dr.tobytes() and np.array_equal(P, Pr)
