"""Trilinear weights of the table-gradient scatter.  A batch of one ray with one sample
leaves, at each level, dL/dfeat times the 8 corner weights: their ratio to the sum over the
corners (the weights add up to 1) is the weight itself, whatever the MLP's precision.
Reference: the FP64 oracle's weights of the FP32 position.  The offsets in a cell are exact
in FP32 and 1 - w is rounded once, so a weight is off by its two products, the product with
dL/dfeat and at most three such roundings, and the sum of the corners by as much: 12 x 2^-24
relative (times the sum of the weights' magnitudes, which is 1 inside the unit cube), for
positions in the first cell of an axis (where the weight of the upper vertex is the
position's own tiny offset) as anywhere else."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = 12 * 2.0 ** -24
POINTS = [(1.3e-6, 0.37, 2.7e-5),   # the first cell in x and z: offsets of 1e-5 and less
          (0.61, 4.1e-6, 0.83),     # in y
          (0.29, 0.71, 0.453),      # inside
          (0.99987, 0.0311, 0.5)]   # the last cell; at a vertex of every level


@pytest.mark.parametrize("prec", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("box", [1.0, 1.4])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_corner_weights(prec, box, axis):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2210_13641_gb300 import NerfMap, pack_params
    cfg = synth.config_small(precision=prec, occ_res=0, n_levels=9, log2_table=12, n_min=4, growth=1.6,
                             max_samples=1, n_steps=1, box_max=np.full(3, box, np.float32))
    P = synth.random_params(cfg, 5, table_scale=0.02, mlp_std=0.3)
    res = oracle.level_resolutions(cfg)
    points = POINTS + ([(1.06, 1.0e-5, 1.03)] if box > 1 else [])
    m = NerfMap(cfg, occ_every=0)
    m.set_params(pack_params(P))
    for i, point in enumerate(points):
        kf = synth.c1_keyframe(i, W=1, H=1)
        d = np.eye(3, dtype=np.float32)[axis]             # the camera looks along the axis
        R = np.stack([np.roll(d, 1), np.roll(d, 2), d], axis=1)
        o = np.array(point, np.float32)
        o[axis] = np.float32(np.float32(point[axis]) - np.float32(cfg.near))
        kf.c2w = np.concatenate([R, o[:, None]], axis=1).astype(np.float32)
        kf.kf_id = 0
        m.add_keyframe(kf)                                # replaces the one before
        m.step(1, seed=3, no_update=True)
        G = m.unpack(m.get_grads())["tables"].astype(np.float64)
        ref = oracle.forward_backward(cfg, P, [kf], 1, 3, 0)
        assert len(ref["t"]) == m.stats().n_samples == 1
        _, idx, wts = oracle.hash_encode(cfg, res, P["tables"], ref["x"])
        for l in range(cfg.n_levels):
            slots, inv = np.unique(idx[0, l], return_inverse=True)
            w = np.bincount(inv, weights=wts[0, l])
            for f in range(2):
                g = G[l, slots, f]
                assert g.sum() != 0.0
                assert np.all(np.abs(g / g.sum() - w) <= TOL * np.abs(w) * np.abs(w).sum()), (i, l, f, g / g.sum(), w)
    m.close()
