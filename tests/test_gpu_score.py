"""vbgs_elbo and vbgs_reassign: the tensor-core score lists against the dense
launch (VBGS_FLAG_NO_SKIP), the posterior they read after other calls, and the
selection of reassign against a plain sort.

Tolerances: a term the lists leave out is below e^-37 / K of its point's sum,
so FP32 sums and merges do not change (one unit in the last place, 1.2e-7, only
where a sum lies within 1e-16 of a rounding boundary): 1e-12 on the lse.  The
selection orders 64-bit keys and indices: equal.
"""
from __future__ import annotations

import numpy as np
import pytest

from oracle import oracle as O
from paper_2603_08499_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def V():
    from paper_2603_08499_gb300 import build
    build.build()
    from paper_2603_08499_gb300 import vbgs
    return vbgs


@pytest.mark.parametrize("form", ["fp16x3", "bf16x3"])
@pytest.mark.parametrize("N,K", [(1, 1), (127, 129), (129, 64), (1_000, 3_000), (4_097, 640)])
def test_lists_equal_dense(V, form, N, K):
    X, pr = synth.c1_workload(seed=N + K, N=N, K=K)
    S = O.cavi_frame(X, pr, np.zeros((K, 28)), 2)[1]
    out = []
    for flags in (0, V.VBGS_FLAG_NO_SKIP):
        m = V.Model(pr, form, flags=flags)
        m.set_stats(S)
        e, lse = m.elbo(X, want_lse=True)
        out.append((e, lse))
        m.close()
    assert O.relerr(out[0][1], out[1][1]) <= 1e-12
    assert O.relerr(out[0][0], out[1][0]) <= 1e-12


def test_room_lists_equal_dense(V):
    room = synth.Room(seed=12)
    pr = synth.room_prior(20_000, seed=12)
    X = [synth.room_frame(t, seed=12, width=100, height=100, room=room) for t in range(3)]
    m = V.Model(pr, "fp16x3")
    m.update(X[0], 3)
    m.update(X[1], 3)
    S = m.stats()
    out = []
    for flags in (0, V.VBGS_FLAG_NO_SKIP):
        d = V.Model(pr, "fp16x3", flags=flags)
        d.set_stats(S)
        out.append(d.elbo(X[2], want_lse=True))
        d.close()
    m.close()
    assert O.relerr(out[0][1], out[1][1]) <= 1e-12


@pytest.mark.parametrize("form", ["fp64", "fp32", "fp16x3"])
def test_posterior_read_after_other_calls(V, form):
    """The posterior vbgs_elbo reads is prior0 (+) S_past whatever ran before:
    the same value as a context that was only given those statistics (the
    components' order differs, so sums agree to the form's rounding)."""
    room = synth.Room(seed=13)
    pr = synth.room_prior(1_500, seed=13)
    X = [synth.room_frame(t, seed=13, width=64, height=64, room=room) for t in range(4)]
    tol = {"fp64": 1e-11, "fp32": 1e-5, "fp16x3": 1e-4}[form]
    g = np.random.default_rng(0).gumbel(size=X[2].shape[0])

    def fresh(S, m0):
        d = V.Model({**pr, "m0": m0}, form)
        d.set_stats(S)
        e, lse = d.elbo(X[3], want_lse=True)
        d.close()
        return e, lse

    m = V.Model(pr, form)
    m0 = pr["m0"].copy()

    def check():
        e, lse = m.elbo(X[3], want_lse=True)
        e_ref, lse_ref = fresh(m.stats(), m0)
        assert O.relerr(e, e_ref) <= tol and O.relerr(lse, lse_ref) <= tol
        assert m.elbo(X[3]) == e

    m.update(X[0], 2)
    check()
    m.update(X[1], 2)
    check()
    pts, comps = m.reassign(X[2], 20, g)
    m0[comps] = X[2][pts]
    check()
    m.update(X[2], 1)
    check()
    m.set_stats(m.stats() * 0.5)
    check()
    bad = X[3].copy()
    bad[5, 1] = np.nan
    with pytest.raises(V.VbgsError) as err:
        m.elbo(bad)
    assert err.value.code == V.VBGS_EINVAL
    check()
    V.vbgs_update_batched([m.ctx], [X[0]], 2)
    check()
    m.update(X[1], 1)
    V.vbgs_update_batched([m.ctx], [X[0]], 2)
    check()
    m.close()


@pytest.mark.parametrize("n", [1, 31, 500, 1_024, 1_025, 2_500])
@pytest.mark.parametrize("ties", ["none", "key", "all"])
def test_selection(V, n, ties):
    """Selected and sorted calls (n at the limit of either) against a plain
    sort: many equal counts, with and without equal tie keys, and equal point
    keys."""
    rng = np.random.default_rng(n)
    K, N = 3_001, 4_099
    X, pr = synth.c1_workload(seed=77, N=N, K=K)
    S = np.zeros((K, 28))
    used = rng.choice(K, 400, replace=False)
    S[used, 0] = rng.integers(1, 4, 400)
    S[used, 1:7] = S[used, :1] * pr["m0"][used]
    u = [(i, j) for i in range(6) for j in range(i, 6)]
    S[used, 7:] = np.stack([S[used, 0] * pr["m0"][used, i] * pr["m0"][used, j] for i, j in u], 1)
    key = {"none": rng.uniform(-1, 1, K), "key": rng.integers(-2, 3, K).astype(float), "all": None}[ties]
    g = rng.gumbel(size=N)
    if ties == "all":
        X = np.repeat(X[: N // 3 + 1], 3, axis=0)[:N].copy()
        g = np.repeat(g[: N // 3 + 1], 3)[:N].copy()
    m = V.Model(pr, "fp64")
    m.set_stats(S)
    lse = m.elbo(X, want_lse=True)[1]
    pts, comps = m.reassign(X, n, g, 1.0, key)
    keys = g - lse
    assert np.array_equal(pts, np.lexsort((np.arange(N), -keys))[:n])
    v = np.zeros(K) if key is None else key
    assert np.array_equal(comps, np.lexsort((np.arange(K), v, S[:, 0]))[:n])
    assert np.array_equal(m.lse(N), lse)
    # a bad value refuses the call and leaves the prior as it is
    before = m.posterior()["m"]
    bad = g.copy()
    bad[-1] = np.inf
    with pytest.raises(V.VbgsError) as err:
        m.reassign(X, n, bad, 1.0, key)
    assert err.value.code == V.VBGS_EINVAL
    if key is not None:
        bk = key.copy()
        bk[0] = np.nan
        with pytest.raises(V.VbgsError):
            m.reassign(X, n, g, 1.0, bk)
    assert np.array_equal(m.posterior()["m"], before)
    e0 = m.elbo(X)
    m.close()
    m0 = pr["m0"].copy()
    m0[comps] = X[pts]
    d = V.Model({**pr, "m0": m0}, "fp64")
    d.set_stats(S)
    assert O.relerr(d.elbo(X), e0) <= 1e-12
    d.close()

