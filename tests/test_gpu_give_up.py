"""GPU tests (-m gpu): solves whose waits run out at any point, on all warps of a
CTA or on some, end with FW_ERR_TIMEOUT (or in time), and the stream's next solve
is right."""
from __future__ import annotations

import numpy as np
import pytest

from fwtest import fw, gpu_solve

pytestmark = pytest.mark.gpu


# (limits around the waits of such a solve, 20 to 400 us, and below any; a wait
# looks at the clock every 16 polls, so that the warps of a CTA differ)
@pytest.mark.parametrize("limit_ns", [1, 60_000, 330_000, 400_000])
@pytest.mark.parametrize("dtype,bs", [(np.int32, 64), (np.int32, 128), (np.float32, 64),
                                      (np.float32, 128), (np.float64, 64), (np.int64, 64)])
def test_short_limits_end(dtype, bs, limit_ns):
    import torch
    m = fw()
    n = 20 * bs + 5
    r = np.random.RandomState(bs)
    W = (1 + r.randint(0, 2000, (n, n))).astype(dtype)
    np.fill_diagonal(W, 0)
    full = torch.zeros((n, m.padded(n)), dtype=torch.from_numpy(W).dtype, device="cuda")
    full[:, :n] = torch.from_numpy(W).cuda()
    for _ in range(3):
        D = full.clone()[:, :n]
        P = torch.zeros((n, full.shape[1]), dtype=torch.int32, device="cuda")[:, :n]
        m.fw_solve_ex(D, P, m.Options.default(bs=bs, timeout_ns=limit_ns))
        try:
            m.fw_sync_status()
        except m.FWError as e:
            assert e.code == 3
    Dg, Pg = gpu_solve(W, bs=bs)
    Dr, Pr = gpu_solve(W, bs=bs, driver=2)
    assert Dg.tobytes() == Dr.tobytes() and np.array_equal(Pg, Pr)
