"""The sparse-first-layer LBF kernel over its tile sizes: 32 rows (both agents' hidden layers
staged at once, the agents on different tensor-memory lanes), up to 64 and up to 128, one
and two rows per warp slot (128- and 64-wide layers), a stage of 32 rows at a time (fp32
128 x 128 on 12x11, where shared memory has room for no more), contiguous, gathered and
rule-teammate tiles, ragged last ones.  Along the kernel's own actions: observations,
rewards and dones bit for bit, log-probabilities and values within the usual tolerance."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_util import close, require_gpu
from paper_2609_13716_gb300 import aht, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height,hidden,dtype,n,pool", [
    (12, 12, (128, 128), "bf16", 203, [1]),         # 32-row tiles
    (12, 12, (128, 128), "bf16", 4900, [1]),        # 64-row tiles, contiguous
    (12, 12, (128, 128), "bf16", 9800, [1, 2, 3]),  # 128-row tiles, gathered
    (8, 9, (64, 64), "f32", 9900, [1]),             # two rows per slot, 128-row tiles
    (9, 8, (64, 128), "bf16", 301, [1, -3]),        # a rule teammate; other widths
    (11, 12, (128, 128), "f32", 9750, [1, 2]),      # a 32-row stage, 128-row tiles
])
def test_tiles(width, height, hidden, dtype, n, pool):
    require_gpu()
    T = 3
    env = W.EnvSpec(kind=W.LBF, width=width, height=height, n_food=3, max_agent_level=3, episode_len=2)
    rng = np.random.Generator(np.random.Philox(n))
    n_pol = 1 + max(pool)
    pop = []
    for p in range(n_pol):
        dims = [env.obs_dim, *hidden, env.n_actions + (1 if p == 0 else 0)]
        layers = [tuple((rng.standard_normal(s) * 0.1).astype(np.float32) for s in ((dims[i + 1], dims[i]), (dims[i + 1],)))
                  for i in range(3)]
        pop.append([tuple(W.round_to_bf16(x) for x in l) for l in layers] if dtype == "bf16" else layers)
    to = torch.bfloat16 if dtype == "bf16" else torch.float32
    tpop = [[(torch.from_numpy(w).to(to), torch.from_numpy(b).to(to)) for w, b in p] for p in pop]
    ctx = aht.aht_create(env, tpop, n, 9, has_value_head=[1] + [0] * (n_pol - 1),
                         weight_dtype=aht.AHT_BF16 if dtype == "bf16" else aht.AHT_FP32)
    traj = aht.traj_buffers(ctx, T)
    aht.aht_rollout(ctx, 0, pool, T, traj)
    aht.aht_sync(ctx)
    g = {k: v.cpu().numpy() for k, v in traj.items()}
    ids = np.unique(np.r_[0, n - 1, rng.integers(0, n, 400)])  # the oracle plays a sample of the envs
    d = O.env_desc(*env.astuple())
    acts = np.ascontiguousarray(np.stack([g["actions"], g["tm_actions"]], -1)[:, ids])
    ref = O.rollout(d, O.Policies(pop), 9, O.reset_envs(d, 9, ids), 0, T, 0, pool, forced=acts, env_ids=ids, n_threads=8)
    assert ref["rc"] == 0
    for k in ("obs", "rewards", "dones"):
        assert np.array_equal(g[k][:, ids], ref[k]), k
    for k in ("logp", "values"):
        ok, worst = close(g[k][:, ids], ref[k])
        assert ok, f"{k}: {worst:.3g}"
    ok, worst = close(g["last_value"][ids], ref["last_value"])
    assert ok, f"last_value: {worst:.3g}"
    own = ref["own_actions"] != acts
    assert (ref["margin"][own] < 1e-5).all(), "actions away from a CDF edge"
