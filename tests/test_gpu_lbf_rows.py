"""Observation rows that the two-group LBF kernel moves cell by cell from step to step, bit
for bit against the oracle along the same actions, through eaten foods and resets: the
smallest grid (rows of 9 words, one tensor-memory chunk per half or none), odd ones, and the
widest that fits (63 cells: the constant input is the operand's last column); one to three
foods; contiguous and gathered tiles, the last one ragged; and seat 1's rows (IPPO)."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import require_gpu
from paper_2609_13716_gb300 import aht, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,n_food", [(3, 3, 1), (3, 4, 2), (5, 6, 3), (7, 9, 3), (9, 7, 1)])
@pytest.mark.parametrize("pool", [1, 3])
def test_rows_follow_the_state(width, height, n_food, pool):
    require_gpu()
    N, T, H = 203, 45, 64
    env = W.EnvSpec(kind=W.LBF, width=width, height=height, n_food=n_food, max_agent_level=2, episode_len=17)
    rng = np.random.Generator(np.random.Philox(100 * width + height))
    dims = [env.obs_dim, H, H, env.n_actions]
    pop = []
    for p in range(pool + 1):
        layers = []
        for i in range(3):
            out = dims[i + 1] + (1 if i == 2 and p < 2 else 0)
            layers.append(tuple(W.round_to_bf16((rng.standard_normal(s) * 0.1).astype(np.float32))
                                for s in ((out, dims[i]), (out,))))
        pop.append(layers)
    tpop = [[(torch.from_numpy(w).bfloat16(), torch.from_numpy(b).bfloat16()) for w, b in p] for p in pop]
    heads = [1, 1] + [0] * (pool - 1)
    ctx = aht.aht_create(env, tpop, N, 5, has_value_head=heads, weight_dtype=aht.AHT_BF16)
    traj = aht.traj_buffers(ctx, T)
    seat1 = {k: v for k, v in aht.traj_buffers(ctx, T).items() if k != "teammate"}
    ids = list(range(1, 1 + pool))
    if pool == 1:
        aht.aht_rollout_ippo(ctx, 0, 1, T, traj, seat1)
    else:
        aht.aht_rollout(ctx, 0, ids, T, traj)
    aht.aht_sync(ctx)
    d = O.env_desc(*env.astuple())
    acts = torch.stack([traj["actions"], traj["tm_actions"]], -1).cpu().numpy()
    ref = O.rollout(d, O.Policies(pop), 5, O.reset_all(d, 5, N), 0, T, 0, ids, forced=acts)
    assert ref["rc"] == 0
    assert ref["dones"].any() and (ref["rewards"] > 0).any()
    assert np.array_equal(traj["obs"].cpu().numpy(), ref["obs"])
    assert np.array_equal(traj["rewards"].cpu().numpy(), ref["rewards"])
    assert np.array_equal(traj["dones"].cpu().numpy(), ref["dones"])
    if pool == 1:
        assert np.array_equal(seat1["obs"].cpu().numpy(), ref["obs_tm"])
