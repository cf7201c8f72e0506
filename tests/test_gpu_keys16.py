"""GPU tests (-m gpu) of the int32 solver's 16-bit packed keys: weights on both
sides of the bounds that choose between 16-bit keys, 32-bit keys and compare
and select, with and without missing edges, whole and ragged tiles, and
matrices whose tiles are of both kinds, against the full oracle."""
from __future__ import annotations

import numpy as np
import pytest

import graphgen
import oracle
from fwtest import INF, check_int_full, gpu_solve

pytestmark = pytest.mark.gpu


def _check(W, bs, **kw):
    D, P = gpu_solve(W, bs=bs, **kw)
    Do, Po = oracle.fw_i64(W)
    check_int_full(W, D, P, Do, Po, oracle.path_count_i64(W, Do))


# BS = 128 / 64 / 32: sums of two panel bounds below 511 / 1023 / 2047 (255 /
# 511 / 1023 beside a missing edge) take 16-bit keys
@pytest.mark.parametrize("bs,n", [(32, 97), (32, 160), (64, 200), (64, 320), (128, 385), (128, 512)])
@pytest.mark.parametrize("hi", [1, 60, 300, 2500, 100000])
@pytest.mark.parametrize("p", [0.02, 1.0])
def test_weights_across_the_bounds(bs, n, hi, p):
    _check(graphgen.dense_graph_i32(n, seed=bs + hi, p=p, lo=1, hi=hi), bs, extra_ld=4)


@pytest.mark.parametrize("bs", [32, 64, 128])
@pytest.mark.parametrize("far", [300, 3000, 10**6])
def test_tiles_of_both_kinds(bs, far):
    """Every other tile row and column holds a vertex far from all others: its
    tiles exceed the 16-bit bounds (10^6 at BS = 128 with the far pairs' sums:
    the 32-bit ones too), so remaining tiles meet operands of both kinds."""
    n = 4 * bs + 3
    W = graphgen.dense_graph_i32(n, seed=far, p=0.6, lo=1, hi=40)
    for v in range(bs // 2, n, 2 * bs):
        W[v, :] = np.where(np.arange(n) % 3 == 0, far, INF)
        W[:, v] = np.where(np.arange(n) % 2 == 0, 2 * far, INF)
        W[v, v] = 0
    _check(W, bs)


@pytest.mark.parametrize("bs", [32, 64, 128])
def test_distance_only_and_unit_weights(bs):
    n = 3 * bs + 5
    W = graphgen.dense_graph_i32(n, seed=9, p=0.05, lo=1, hi=1)
    _check(W, bs, lookahead=0)
    import torch
    import paper_2403_18619_gb300 as fw
    D, P = fw.solve(torch.from_numpy(W).cuda(), fw.Options.default(bs=bs), with_pred=False)
    assert P is None
    assert np.array_equal(D.cpu().numpy().astype(np.int64), oracle.fw_i64(W)[0])
