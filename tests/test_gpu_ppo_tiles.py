"""The gradient kernel's tiles against the fp64 oracle at the sizes where its split can go
wrong: one tile, fewer tiles than SMs, one more than the SMs of a GB300 (one CTA runs two),
two rounds plus one; the narrowest and widest observation rows (the constant-1 column in the
first and the last words of the padded width) and output counts.  Random trajectories with
byte observations; the old values lie outside the clip band on either side of the new ones
(inside it the two value losses are equal and rounding picks the branch).  The tolerance is
that of test_gpu_ppo.py, from the same arithmetic."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2609_13716_gb300 import aht
from gpu_util import require_gpu
from test_gpu_ppo import check_grad, check_stats, hp_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,A,tiles", [(4, 2, 1), (100, 6, 3), (144, 7, 153), (204, 3, 305), (196, 6, 152)])
def test_gradient_over_tiles_and_widths(D, A, tiles):
    require_gpu()
    rng = np.random.default_rng(1000 * tiles + D)
    S = 64 * tiles
    layers = [(rng.normal(0, 1 / np.sqrt(i), (o, i)).astype(np.float32), rng.normal(0, 0.1, o).astype(np.float32))
              for i, o in ((D, 128), (128, 128), (128, A + 1))]
    b = dict(obs=rng.integers(0, 3, (1, S, D)).astype(np.uint8), actions=rng.integers(0, A, (1, S)).astype(np.uint8),
             logp=(-np.log(A) + rng.normal(0, 0.2, (1, S))).astype(np.float32),
             values=rng.choice([-4.0, 4.0], (1, S)).astype(np.float32),
             advantages=rng.normal(0, 1, (1, S)).astype(np.float32),
             targets=rng.normal(0, 0.5, (1, S)).astype(np.float32))
    L = aht.aht_learner_create(D, A, [(torch.from_numpy(w), torch.from_numpy(x)) for w, x in layers], epochs=1,
                               minibatches=1, seed=7)
    g = torch.empty(L.n_params, device="cuda")
    st = torch.empty(6, device="cuda")
    aht.aht_ppo_grad(L, {k: torch.from_numpy(v).cuda() for k, v in b.items()}, 0, 0, g, st)
    aht.aht_learner_sync(L)
    net = O.ppo_net(D, 128, 128, A)
    p0 = O.flat_params([(w.astype(np.float64), x.astype(np.float64)) for w, x in layers])
    go, so = O.ppo_grad(net, p0, O.PpoBatchNp(**b), O.perm(7, 0, S), hp_of(L, epoch0=0), n_threads=8)
    check_grad(g.cpu().numpy().astype(np.float64), go, net)
    check_stats(st.cpu().numpy().astype(np.float64), so, S)
