"""The sparse CUDA-core passes (pairs above e^-(ln K + 37) of a point's mass)
against the dense ones (VBGS_FLAG_NO_SKIP) on the same points and components in
the same order, one E-step from the same state.

Tolerances, derived from the arithmetic:
* FP64: a point loses at most K e^-(ln K + 37) = 8.5e-17 of its mass; the sums
  take the same terms in another order, off by at most ~sqrt(n) 2^-53 for n <=
  20,000 positive terms (1.6e-14), and a logit carries a few roundings of its
  largest term (|q| up to ~1e4 near the outliers: 1e-12).
* FP32: the same operations in the same order over the terms that reach FP32
  rounding.  Only a term within 1e-16 of a rounding boundary can move a sum, by
  one unit in the last place (2^-23); four of them bound a whole array.
"""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_08499_gb300 import synth

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-12, "fp32": 4 * 2.0 ** -23}


@pytest.fixture(scope="module")
def V():
    from paper_2603_08499_gb300 import build
    build.build()
    from paper_2603_08499_gb300 import vbgs
    return vbgs


def both(V, X, prior, form, S, split=0):
    out = []
    for flags in (V.VBGS_FLAG_NO_REORDER, V.VBGS_FLAG_PLAIN):
        m = V.Model(prior, form, flags=flags | split)
        m.set_stats(S)
        e, lse0 = m.elbo(X, want_lse=True)
        tr = m.update(X, 1)
        out.append((np.array([e, tr[0]]), lse0, m.lse(X.shape[0]), m.frame_stats()))
        m.close()
    return out


def agree(V, X, prior, form, S, split=0):
    sparse, dense = both(V, X, prior, form, S, split)
    for i, (a, b) in enumerate(zip(sparse, dense)):
        assert np.all(np.isfinite(a)), i
        assert O.relerr(a, b) <= TOL[form], (i, O.relerr(a, b))


@pytest.mark.parametrize("form", ["fp64", "fp32"])
@pytest.mark.parametrize("N,K", [(1, 1), (31, 33), (32, 32), (33, 31), (1023, 5), (1025, 257), (2500, 64), (300, 2440),
                                 (3000, 2431), (20000, 17)])
def test_sizes(V, form, N, K):
    X, pr = synth.c1_workload(seed=N + K, N=N, K=K)
    S = np.zeros((K, 28))
    agree(V, X, pr, form, S)
    m = V.Model(pr, "fp64")
    m.update(X, 2)
    S = m.stats()
    m.close()
    agree(V, X, pr, form, S)


@pytest.mark.parametrize("form", ["fp64", "fp32"])
def test_room_and_far_points(V, form):
    """Thin components, and points far from every component: their largest
    logit is thousands of nats below the others' and the seed can be poor."""
    room = synth.Room(seed=6)
    pr = synth.room_prior(4_000, seed=6)
    X = synth.room_frame(1, seed=6, width=64, height=64, room=room)
    m = V.Model(pr, "fp64")
    m.update(synth.room_frame(0, seed=6, width=64, height=64, room=room), 3)
    S = m.stats()
    m.close()
    agree(V, X, pr, form, S)
    agree(V, X, pr, form, S, split=V.VBGS_FLAG_SPLIT)
    Y = X.copy()
    rng = np.random.default_rng(3)
    far = rng.choice(Y.shape[0], 40, replace=False)
    Y[far, :3] += rng.uniform(-12.0, 12.0, (40, 3))
    agree(V, Y, pr, form, S)


@pytest.mark.parametrize("form", ["fp64", "fp32"])
def test_unordered_points(V, form):
    """Caller's order without any locality: the boxes rule out nothing."""
    X, pr = synth.c1_workload(seed=31, N=4_321, K=613)
    X = X[np.random.default_rng(1).permutation(X.shape[0])]
    agree(V, X, pr, form, np.zeros((613, 28)))
