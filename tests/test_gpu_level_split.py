"""Steps on maps whose tables do not fit the L2, which take their finest levels level by level
in launches of their own (the forward's gathers before it, the scatter after the backward):
that such a step takes this way and a small batch on the same map does not (launches per
phase); and the gradients where test_gpu_tile_scatter.py does not reach: no more than eight
levels (all of them level by level), a box that reaches past the unit cube, and pose
gradients (whose backward keeps all levels and uses the same half of the encoding buffer).
Reference: the FP64 oracle with the MLP's rounding model; relative L2 2e-3, the tensor-core
forms' gradient tolerance (test_gpu_tc.py, test_gpu_pose.py)."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = 2e-3
RAYS, SMAX = 4099, 128            # 524 672 samples at most: just above the rule's 2^19
# (levels, log2 table, growth, box upper corner, pose gradients)
CASES = [(5, 22, 2.6, 1.0, False), (8, 22, 1.9, 1.0, False), (8, 22, 1.9, 1.3, False), (11, 21, 1.6, 1.3, False),
         (10, 21, 1.7, 1.0, True)]


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("prec", ["fp16", "bf16"])
@pytest.mark.parametrize("levels,log2t,growth,box,pose", CASES)
def test_large_tables_level_by_level(prec, levels, log2t, growth, box, pose):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    if levels * (8 << log2t) <= torch.cuda.get_device_properties(0).L2_cache_size:
        pytest.skip("the tables fit this device's L2")
    from paper_2210_13641_gb300 import NerfMap, pack_params
    cfg = synth.config_small(precision=prec, occ_res=0, n_levels=levels, log2_table=log2t, growth=growth,
                             max_samples=SMAX, step=np.float32(0.03), n_steps=60,
                             box_max=np.full(3, box, np.float32),
                             grid_inv_size=np.float32(1.5 if box > 1 else 1.0))
    P = synth.random_params(cfg, 11, table_scale=0.5, mlp_std=0.15)
    kf = synth.c1_keyframe(12, W=40, H=30)
    m = NerfMap(cfg, occ_every=0)
    m.set_params(pack_params(P))
    m.add_keyframe(kf)
    for rays, split in ((1021, 0), (RAYS, 1)):
        m.profile(True)
        loss = m.step(rays, seed=3, no_update=True, pose_grad=pose)
        ph = m.profile_read()
        m.profile(False)
        assert ph["field_fwd"]["launches"] == 1 + split
        # a pose step: the backward, which takes all levels itself, and the sums along the rays
        assert ph["field_bwd"]["launches"] == (2 if pose else 1 + split)
    G = m.unpack(m.get_grads())
    g_pose = m.pose_grads() if pose else None
    m.close()
    ref = oracle.forward_backward(cfg, P, [kf], RAYS, 3, 0, mlp_bits=prec)
    assert loss == pytest.approx(ref["loss"], rel=TOL)
    for k, g in ref["grads"].items():
        assert _rel(G[k], g) <= TOL, k
    if pose:
        assert _rel(g_pose, oracle.pose_gradients(cfg, P, [kf], RAYS, 3, 0, mlp_bits=prec)["pose_grads"]) <= TOL
