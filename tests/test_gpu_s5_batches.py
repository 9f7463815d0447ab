"""aht_s5_step over batch sizes that change its output tiles (narrow ones down to 32 columns for
a batch of few row tiles, full-width ones for many) and its last row tile (one row, a row
block's edge, a full tile and one row more), on one handle, against the fp64 oracle on a
sample of the rows (rows are independent)."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import close, np_, require_gpu
from paper_2609_13716_gb300 import aht, workloads as W

pytestmark = pytest.mark.gpu


def test_batches_of_one_handle():
    require_gpu()
    K, A, P = 52, 6, 64
    params = W.s5_params(11, K, A, H=128, P=P, F=256)
    pol = aht.aht_s5_create(params, 2600)
    net = O.S5(params)
    rng = np.random.default_rng(1)
    for n in (2600, 1, 8, 9, 128, 129, 640, 1):  # a small batch after a large one reads no stale row
        obs = rng.integers(0, 4, (n, K)).astype(np.uint8)
        state0 = (0.3 * rng.standard_normal((n, 2 * P))).astype(np.float32)
        rows = np.unique(np.r_[0, n - 1, rng.integers(0, n, 20)])
        state, ref = torch.from_numpy(state0).cuda(), state0[rows].astype(np.float64)
        logits, values = torch.empty(n, A, device="cuda"), torch.empty(n, device="cuda")
        for t in range(2):  # the second step continues the state the first one wrote
            reset = (rng.random(n) < 0.3).astype(np.uint8)
            legal = (rng.random((n, A)) < 0.7).astype(np.uint8)
            legal[:, 0] = 1
            aht.aht_s5_step(pol, torch.from_numpy(obs).cuda(), torch.from_numpy(reset).cuda(), state, logits, values,
                            torch.from_numpy(legal).cuda())
            aht.aht_s5_sync(pol)
            lg, v = net.step(obs[rows], reset[rows], ref, legal[rows])
            on = legal[rows] == 1
            for name, got, want in (("logits", np_(logits)[rows][on], lg[on]), ("values", np_(values)[rows], v),
                                    ("state", np_(state)[rows], ref)):
                ok, worst = close(got, want)
                assert ok, f"{name}, n = {n}, step {t}: {worst:.3g}"
    pol.close()
