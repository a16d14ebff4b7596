"""map_marginal_covariances over the block structures a pixel may have: one to eight blocks
per pixel, unused ones (-1), two blocks of one pose, poses that change at every pixel, one
keyframe and the largest window; against the FP64 oracle within 1e-9 relative (FP64 on
both sides, other summation orders, as test_gpu_covariance.py)."""

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _window(K, p, B, seed, shuffle, repeat):
    rng = np.random.default_rng(seed)
    blk = np.full((p, B), -1, np.int32)
    e = rng.normal(size=(p, B, 6))
    for q in range(p):
        own = (q * K) // p if not shuffle else int(rng.integers(K))
        r = np.random.default_rng(q if shuffle else own)
        used = int(r.integers(1, B + 1))
        blk[q, :used] = r.integers(0, K, used) if repeat else r.permutation(K)[:used] if K >= used else own
        if not repeat and K < used:
            blk[q, 1:] = -1
    P = rng.uniform(0.5, 3.0, p)
    E = oracle.arrow_dense_E(6 * K, blk, np.where(blk[..., None] >= 0, e, 0.0))
    A = rng.normal(size=(6 * K, 6 * K))
    C = (E / P) @ E.T + A @ A.T + 6 * K * np.eye(6 * K)   # so that the reduced matrix is positive definite
    return C, P, blk, e


@pytest.mark.parametrize("K,p,B,shuffle,repeat", [
    (1, 3, 1, False, False), (2, 37, 2, False, True), (5, 1000, 3, True, False), (7, 2500, 4, True, True),
    (24, 700, 5, False, True), (9, 333, 6, True, True), (12, 900, 7, False, False), (24, 5000, 8, True, True)])
def test_blocks_match_oracle(K, p, B, shuffle, repeat):
    import __graft_entry__
    __graft_entry__.build()
    from paper_2210_13641_gb300.binding import marginal_covariances
    C, P, blk, e = _window(K, p, B, 10 * K + B, shuffle, repeat)
    ST, Sd = marginal_covariances(C, P, blk, e)
    rST, rSd = oracle.marginal_covariances(C, P, blk, np.where(blk[..., None] >= 0, e, 0.0))
    assert np.linalg.norm(ST - rST) <= 1e-9 * np.linalg.norm(rST)
    assert np.allclose(Sd, rSd, rtol=1e-9, atol=0)
