"""The CUDA-core MLP tile at the edges of its row, column and feature handling, through
aht_policy_forward, against a plain fp64 torch forward."""
import numpy as np
import pytest
import torch

from gpu_util import require_gpu
from paper_2609_13716_gb300 import aht, workloads as W

pytestmark = pytest.mark.gpu

ENVS = {"lbf5": W.EnvSpec(kind=W.LBF, width=5, height=5, n_food=3, max_agent_level=3, episode_len=50),
        "kitchen": W.EnvSpec(kind=W.OVERCOOKED, width=5, height=4, episode_len=50, cook_time=20, soup_reward=20),
        "hanabi": W.EnvSpec(kind=W.HANABI), "minihanabi": W.EnvSpec(kind=W.MINI_HANABI)}


def policy(env, h0, h1, seed):
    rng = np.random.Generator(np.random.Philox(seed))
    dims = [env.obs_dim, h0, h1, env.n_actions + 1]
    return [(torch.from_numpy((rng.standard_normal((dims[i + 1], dims[i])) * 0.1).astype(np.float32)),
             torch.from_numpy((rng.standard_normal(dims[i + 1]) * 0.1).astype(np.float32))) for i in range(3)]


def context(env, layers):
    return aht.aht_create(env, [layers], 8, 0, has_value_head=[1], weight_dtype=aht.AHT_FP32)


def forward64(layers, obs):
    h = obs.cpu().double()
    for w, b in layers[:2]:
        h = torch.tanh(h @ w.double().T + b.double())
    return h @ layers[2][0].double().T + layers[2][1].double()


# n: one row, tile edges of 8 and 24 rows, a ragged last tile; hidden widths: the smallest, one
# that is no power of two (a group's threads past the columns), more columns than threads,
# and the widest
@pytest.mark.parametrize("game", list(ENVS))
@pytest.mark.parametrize("hidden", [(16, 48), (272, 80), (512, 512)])
@pytest.mark.parametrize("n", [1, 8, 9, 24, 1217, 3649])
def test_rows_columns_and_features(game, hidden, n):
    require_gpu()
    env = ENVS[game]
    layers = policy(env, *hidden, seed=n)
    ctx = context(env, layers)
    g = torch.Generator().manual_seed(n)
    # bytes of any value; LBF rows list signed 8-bit changes to the empty grid (levels are small)
    top = 128 if game == "lbf5" else 256
    obs = (torch.rand(n, env.obs_dim, generator=g) < 0.3).to(torch.uint8) * \
        torch.randint(1, top, (n, env.obs_dim), generator=g).to(torch.uint8)
    obs[:, env.obs_dim // 2:] = 0          # features no row has
    obs[n // 2] = 0                        # an empty row
    want = forward64(layers, obs)
    out = torch.empty(n, env.n_actions + 1, device="cuda")
    odd = torch.empty(n * env.obs_dim + 1, dtype=torch.uint8, device="cuda")[1:].view(n, env.obs_dim)
    for rows in (obs.cuda(), odd.copy_(obs)):   # word-aligned and unaligned observations
        aht.aht_policy_forward(ctx, 0, rows, out)
        aht.aht_sync(ctx)
        # fp32 sums of up to 660 terms of bytes x 0.1: pre-activations of ~1e2, so 1e-5 before
        # tanh, whose slope is at most 1, and 2e-5 after two more layers of 0.1 weights
        torch.testing.assert_close(out.cpu().double(), want, rtol=1e-4, atol=2e-4)


def test_infinite_weight_of_an_absent_feature_still_gives_nan():
    """0 x inf is NaN in the dense sum, so the listed-features sum must not skip it."""
    require_gpu()
    env = ENVS["kitchen"]
    layers = policy(env, 64, 64, seed=3)
    layers[0][0][5, 7] = float("inf")
    ctx = context(env, layers)
    obs = torch.zeros(4, env.obs_dim, dtype=torch.uint8, device="cuda")
    out = torch.empty(4, env.n_actions + 1, device="cuda")
    aht.aht_policy_forward(ctx, 0, obs, out)
    aht.aht_sync(ctx)
    assert out.isnan().all()
    obs[:, 7] = 1  # inf x 1: tanh(inf) = 1
    aht.aht_policy_forward(ctx, 0, obs, out)
    aht.aht_sync(ctx)
    assert out.isfinite().all()
