"""The backward's gradients (table and weights) at the edges of its 128-sample tiles and of
its 16-sample walks, over dense and hashed levels in every pairing, and for a box that
reaches past the unit cube (samples that extrapolate from the last cell).  Reference: the
FP64 oracle, for the tensor-core forms with the MLP's rounding model; tolerances: relative
L2 2e-3 for those (test_gpu_tc.py's), 1e-4 for the plain FP32 form (a few thousand FP32
terms per sum, and near-kink ReLU branches)."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

# (levels, log2 table, growth, rays, samples per ray, box upper corner)
CASES = [
    (1, 10, 2.0, 1, 24, 1.0),      # one level (hashed or dense alone), a tile of one short ray
    (2, 12, 2.0, 5, 24, 1.0),      # a pair of dense levels
    (5, 10, 1.7, 37, 16, 1.0),     # dense and hashed levels in one warp, truncated rays
    (9, 11, 1.5, 129, 24, 1.0),    # one more than eight levels
    (16, 10, 1.38, 300, 24, 1.0),  # every level, several tiles
    (16, 14, 1.2, 64, 24, 1.0),    # mostly dense levels
    (4, 10, 2.0, 200, 24, 1.3),    # positions up to 1.3: cells clamped to the last one
]


# tables larger than the L2 and enough rays: the finest levels level by level
# (9 levels: one of them as usual; 12: four)
CASES += [(9, 21, 1.9, 4099, 128, 1.0), (12, 21, 1.5, 5000, 128, 1.0)]


@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp32"])
@pytest.mark.parametrize("levels,log2t,growth,rays,smax,box", CASES)
def test_table_gradient_matches_oracle(prec, levels, log2t, growth, rays, smax, box):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2210_13641_gb300 import NerfMap, pack_params
    cfg = synth.config_small(precision=prec, occ_res=0, n_levels=levels, log2_table=log2t, growth=growth,
                             max_samples=smax, step=np.float32(0.03), n_steps=60,
                             box_max=np.full(3, box, np.float32),
                             grid_inv_size=np.float32(1.5 if box > 1 else 1.0))
    P = synth.random_params(cfg, 11, table_scale=0.5, mlp_std=0.15)
    kf = synth.c1_keyframe(12, W=40, H=30)
    m = NerfMap(cfg, occ_every=0)
    m.set_params(pack_params(P))
    m.add_keyframe(kf)
    loss = m.step(rays, seed=3, no_update=True)
    G = m.unpack(m.get_grads())
    m.close()
    ref = oracle.forward_backward(cfg, P, [kf], rays, 3, 0, mlp_bits=prec)
    tol = 1e-4 if prec == "fp32" else 2e-3
    assert loss == pytest.approx(ref["loss"], rel=tol)
    for k, g in ref["grads"].items():
        assert np.linalg.norm(G[k] - g) <= tol * max(np.linalg.norm(g), 1e-30), k
