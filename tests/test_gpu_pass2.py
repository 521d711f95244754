"""The tensor-core statistics pass, whose CTAs each walk several work items:
against the FP64 form from the same state, at one item, fewer items than
resident CTAs, and several items a CTA, within and across component tiles.

Tolerance: as the other comparisons of the hi/lo form with the FP64 form, 1e-3
of the norm of each block of the statistics (22-bit operands on logits of
order 10^2: about 1e-4 in a responsibility), 2e-2 with the 16 bits of the BF16
split (64 times as much).  An item left out or counted
twice is at least 256 of at most 40,000 points: 6e-3.
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
@pytest.mark.parametrize("N,K,dense", [(64, 1, False), (65, 129, True), (9_999, 128, True), (40_000, 300, True),
                                       (40_000, 300, False), (20_000, 5_000, True)])
def test_items_of_a_cta(V, form, N, K, dense):
    X, pr = synth.c1_workload(seed=N + K, N=N, K=K)
    S = []
    for prec in (form, "fp64"):
        m = V.Model(pr, prec, flags=V.VBGS_FLAG_NO_SKIP if dense and prec == form else 0)
        m.update(X, 1)
        S.append(m.frame_stats())
        m.close()
    for sl in (slice(0, 1), slice(1, 7), slice(7, 28)):
        assert O.relerr(S[0][:, sl], S[1][:, sl]) <= (1e-3 if form == "fp16x3" else 2e-2)
