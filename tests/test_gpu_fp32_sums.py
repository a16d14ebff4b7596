"""Weight gradients of the plain FP32 form: how exactly they are summed.

Every ray of a batch is drawn from a keyframe of one pixel and keeps one sample, so all
samples are the same, and the gradient of the batch's mean loss is that of one ray (the
FP64 oracle's).  Adding one value n times in FP32 errs by about n 2^-24 / 9 of the sum
(rms over values; each addition rounds the same way within a binade), so the result tells
the longest chain of additions.  Sums of 128 products, then of a block's tiles (about 216
of 32768), then of the blocks: 2.0e-6 by that model.  One flat sum over a thread's share of
all tiles: 2.5e-5 (16 products a tile) to 9.6e-5 (64).  Tolerance: 1e-5, the suite's bound
for FP32 gradients (test_gpu_parity.py), which also holds the error of one sample's chain.

The second test takes the same bound at the edges of the 128-sample tiles."""

import numpy as np
import pytest

import oracle
import synth
from test_gpu_tile_scatter import CASES

pytestmark = pytest.mark.gpu

REL = 1e-5
WEIGHTS = ("W1", "W2", "W3", "W4", "W5")


def _weight_grads(cfg, P, kf, rays, seed=3):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2210_13641_gb300 import NerfMap, pack_params
    m = NerfMap(cfg, occ_every=0)
    m.set_params(pack_params(P))
    m.add_keyframe(kf)
    m.step(rays, seed=seed, no_update=True)
    n, G = m.stats().n_samples, m.unpack(m.get_grads())
    m.close()
    return n, G


@pytest.mark.parametrize("seed", [1, 2])
def test_equal_samples_sum_like_one(seed):
    rays = 1 << 22
    cfg = synth.config_small(precision="fp32", occ_res=0, max_samples=1)
    P = synth.random_params(cfg, seed, table_scale=0.5, mlp_std=0.3)
    kf = synth.c1_keyframe(seed, W=1, H=1)
    ref = oracle.forward_backward(cfg, P, [kf], 1, 3, 0, magnitudes=True)
    assert len(ref["t"]) == 1 and not ref["near_kink"].any()
    n, G = _weight_grads(cfg, P, kf, rays)
    assert n == rays
    for k in WEIGHTS:
        g = ref["grads"][k]
        assert np.linalg.norm(g) > 0
        assert np.linalg.norm(G[k] - g) <= REL * np.linalg.norm(g), k


@pytest.mark.parametrize("levels,log2t,growth,rays,smax,box", CASES[:7])
def test_weight_gradients_at_tile_edges(levels, log2t, growth, rays, smax, box):
    cfg = synth.config_small(precision="fp32", occ_res=0, n_levels=levels, log2_table=log2t, growth=growth,
                             max_samples=smax, step=np.float32(0.03), n_steps=60,
                             box_max=np.full(3, box, np.float32),
                             grid_inv_size=np.float32(1.5 if box > 1 else 1.0))
    P = synth.random_params(cfg, 11, table_scale=0.5, mlp_std=0.15)
    kf = synth.c1_keyframe(12, W=40, H=30)
    _, G = _weight_grads(cfg, P, kf, rays)
    ref = oracle.forward_backward(cfg, P, [kf], rays, 3, 0)
    for k in WEIGHTS:
        g = ref["grads"][k]
        assert np.linalg.norm(G[k] - g) <= REL * max(np.linalg.norm(g), 1e-30), k
