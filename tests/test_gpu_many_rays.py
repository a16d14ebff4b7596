"""Batches of more than 2^20 rays (a step takes up to 2^24): the sample list is the
oracle's, bit for bit; nothing outside the batch's own buffers is written (another map's
parameters and moments stay as they are); and a view rendered in one piece of more than
2^20 rays (the work buffers have that capacity after such a step) equals the same view
rendered in pieces of 2^18 by a map that has seen no step, bit for bit."""

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

RAYS = (1 << 20) + 4097          # two tiles of 4096 rays more than 2^20, the last of one ray
W, H = 1031, 1021                # 1 052 651 pixels


def _oracle_samples(cfg, kf, seed, step, chunk=1 << 16):
    _, u, v = oracle.draw_rays(seed, step, RAYS, [(kf.W, kf.H)])
    rid, ts = [], []
    for a in range(0, RAYS, chunk):
        n = len(u[a:a + chunk])
        o, d = oracle.cast_rays_f32(np.broadcast_to(kf.c2w, (n, 3, 4)), np.broadcast_to(kf.K, (n, 4)),
                                    u[a:a + chunk], v[a:a + chunk])
        r, _, t, _ = oracle.march(cfg, o, d)
        rid.append((r + a).astype(np.uint32))
        ts.append(t.astype(np.float32))
    return np.concatenate(rid), np.concatenate(ts)


@pytest.mark.parametrize("prec", ["fp16", "fp32"])
def test_more_than_2_20_rays(prec):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2210_13641_gb300 import NerfMap, pack_params
    # up to 40 samples of a ray: more than a render's first pass takes
    cfg = synth.config_small(precision=prec, occ_res=0, max_samples=40, step=np.float32(0.011), n_steps=60)
    P = synth.random_params(cfg, 11, table_scale=0.5, mlp_std=0.15)
    kf = synth.c1_keyframe(12, W=40, H=30)
    other, whole = NerfMap(cfg, occ_every=0), NerfMap(cfg, occ_every=0)
    for m in (other, whole):
        m.set_params(pack_params(P))
        m.add_keyframe(kf)
    whole.step(RAYS, seed=3, no_update=True)
    assert whole.stats().n_rays == RAYS
    rid, t = whole.samples()
    ref_rid, ref_t = _oracle_samples(cfg, kf, 3, 0)
    assert np.array_equal(rid, ref_rid) and np.array_equal(t.view(np.uint32), ref_t.view(np.uint32))
    assert np.bincount(rid, minlength=RAYS).max() > 32
    K = np.array([500.0, 500.0, W / 2, H / 2], np.float32)
    one = whole.render(kf.c2w, K, W, H)
    pieces = other.render(kf.c2w, K, W, H)
    for a, b in zip(one, pieces):
        assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    assert np.isfinite(one[0]).all() and one[2].max() > 0.1
    assert np.array_equal(other.get_params(), pack_params(P))
    assert not any(np.any(x) for x in other.get_adam())
    whole.close()
    other.close()
