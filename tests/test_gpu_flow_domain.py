"""Rows outside of [0,1)^D in the density direction: no access outside of the row's own
logits, whatever the coordinate's value, and no effect on the rows beside them."""
import numpy as np
import pytest

from oracle import flow as FL
from paper_2409_07148_gb300.flowinit import init_flow_params

pytestmark = pytest.mark.gpu

K, E = FL.K, FL.E


def _flow(D, seed, sd=0.1):
    perm, w = init_flow_params(D, seed)
    tail = D // 2 * K * FL.H + D // 2 * K
    w[:, -tail:] = np.random.default_rng(seed + 100).normal(0.0, sd, (w.shape[0], tail)).astype(np.float32)
    return perm, w


def _log_density(perm, w, x):
    """The flow's density direction continued below 0: bin trunc(t K) < 0 lies below
    every bin and has the floor's mass E / K, as has each of the bins 0 .. b between."""
    x = np.array(x, np.float64, copy=True)
    n, D = x.shape
    A = D // 2
    lq = np.zeros(n)
    for l in range(len(perm)):
        ca, cb = perm[l][:A], perm[l][A:]
        Q = FL.bins(w[l], x[:, ca], D)
        t = x[:, cb]
        b = np.minimum(np.trunc(t * K), K - 1).astype(np.int64)
        at = np.maximum(b, 0)[..., None]
        cum = np.concatenate([np.zeros((n, A, 1)), np.cumsum(Q, axis=2)], axis=2)
        qb = np.where(b < 0, E / K, np.take_along_axis(Q, at, axis=2)[..., 0])
        lo = np.where(b < 0, b * E / K, np.take_along_axis(cum, at, axis=2)[..., 0])
        x[:, cb] = lo + (t * K - b) * qb
        lq += np.log(K * qb).sum(axis=1)
    return lq


# 300 rows: two full tiles and a ragged one.  D = 2 and 32 are the ends of the range, where the
# row's tile is first and last in shared memory.
@pytest.mark.parametrize("D", [2, 8, 22, 32])
def test_density_rows_outside_the_cube(D):
    import torch
    from paper_2409_07148_gb300 import jr
    perm, w = _flow(D, 90 + D)
    f = jr.Flow(D, perm, w)
    rng = np.random.default_rng(D)
    x = rng.random((300, D)).astype(np.float32)
    clean = f.log_density(torch.from_numpy(np.ascontiguousarray(x.T)).cuda()).cpu().numpy()
    bad = x.copy()
    values = [-2.0 ** -4, -0.5, -1.0, -17.25, -1e9, -3e38, -np.inf, np.inf, np.nan, 1.0, 2.0, 1e9]
    rows = {}
    for k, v in enumerate(values):  # one coordinate of a row, and a whole row
        for r, d in ((5 + 16 * k, int(rng.integers(D))), (7 + 16 * k, slice(None))):
            bad[r, d] = v
            rows[r] = v
    got = f.log_density(torch.from_numpy(np.ascontiguousarray(bad.T)).cuda()).cpu().numpy()
    assert f.status() == 0
    inside = np.setdiff1d(np.arange(300), list(rows))
    assert np.array_equal(got[inside], clean[inside])
    # moderate values: the continuation's density.  One coordinate's terms are below 7 in magnitude, so
    # FP32 rounds each to 2^-22, 96 at most; a bf16 edge or a bin's edge may go the other way (module
    # test_gpu_flow), which moves a row by the steps of the bf16 roundings: 0.05 is far below a bin's
    # log E = -6.9 and above those.
    small = [r for r, v in rows.items() if np.isfinite(v) and abs(v) <= 2.0]
    want = _log_density(perm, w, bad[small].astype(np.float64))
    assert np.all(np.abs(got[small] - want) <= 0.05), np.abs(got[small] - want).max()


# a batch below one tile and one of three; rows below 0 in one coordinate, or in all of them
@pytest.mark.parametrize("D,rows", [(2, 40), (8, 150)])
def test_training_rows_below_zero(D, rows):
    """The training loss continues bin 0 to coordinates below it: finite, and the
    continuation's value.  The gradient stays finite."""
    import torch
    from paper_2409_07148_gb300 import jr
    perm, w = _flow(D, 60 + D)
    rng = np.random.default_rng(D)
    x = rng.random((rows, D)).astype(np.float32)
    for k, v in enumerate([-2.0 ** -4, -0.5, -1.0, -17.25]):
        x[3 + 8 * k, int(rng.integers(D))] = v
        x[4 + 8 * k] = v
    wt = (rng.random(rows) + 0.05).astype(np.float32)
    loss, g = jr.Flow(D, perm, w).gradient(torch.from_numpy(np.ascontiguousarray(x.T)).cuda(),
                                           torch.from_numpy(wt).cuda())
    y, lq, A = x.astype(np.float64), np.zeros(rows), D // 2
    for l in range(len(perm)):
        ca, cb = perm[l][:A], perm[l][A:]
        Q = FL.bins(w[l], y[:, ca], D)
        t = y[:, cb]
        b = np.minimum(np.trunc(t * K), K - 1).astype(np.int64)
        at = np.maximum(b, 0)[..., None]
        cum = np.concatenate([np.zeros((rows, A, 1)), np.cumsum(Q, axis=2)], axis=2)
        qb = np.take_along_axis(Q, at, axis=2)[..., 0]
        y[:, cb] = np.take_along_axis(cum, at, axis=2)[..., 0] + (t * K - b) * qb
        lq += np.log(K * qb).sum(axis=1)
    want = -(wt * lq).sum() / wt.sum()
    assert abs(loss - want) <= 1e-3 * max(1.0, abs(want)), (loss, want)  # test_gpu_flow_train's bound
    assert np.isfinite(g).all()
