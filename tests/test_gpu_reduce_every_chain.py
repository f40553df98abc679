"""Every chain counts: the reduction with weights of one order against numpy.

With log W within 1 of each other and a distinct R_ee^2, R_g^2 per chain, leaving
out, repeating or swapping any chain moves a sum by at least 1 / (50 n) of it
(n <= 4100), far beyond the tolerance of 4 n 2^-53 plus the weights' own errors.
Real-space, lattice and athermal lattice (weights from counts) inputs at the edges
of quarters, tiles and the merging block; both standard errors.
"""
import math

import numpy as np
import pytest
import torch

from paper_1704_04381_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosen():
    pkg_build.build()
    from paper_1704_04381_gb300 import rosen as r
    r.load()
    return r


@pytest.mark.parametrize("kind", ["space", "lattice", "counts"])
@pytest.mark.parametrize("C", [2, 127, 128, 129, 511, 512, 513, 1537, 2047, 2048, 2049, 4100])
def test_sums(rosen, C, kind):
    g = np.random.default_rng(C)
    N = 9
    lw = g.random(C).astype(np.float32)
    r2, n2 = g.permutation(C) + 1 + C, g.permutation(C) + 1 + C
    inp = dict(N=N, k=7, use_counts=0, C=C)
    if kind == "space":
        dev = dict(logw=lw, r2_f=r2.astype(np.float32), rg2_f=n2.astype(np.float32))
        inp.update(kind=rosen.ROSEN_REDUCE_OFFLATTICE)
        lw, a, b = lw.astype(float), r2.astype(float), n2.astype(float)
    else:
        counts = np.zeros((C, 8), np.uint16)
        counts[:, 2:7] = g.integers(0, 3, (C, 5))
        dev = dict(logw=lw, r2_i=r2.astype(np.int32), n2rg2=n2.astype(np.int64),
                   counts=counts)
        inp.update(kind=rosen.ROSEN_REDUCE_LATTICE, k=0)
        a, b, lw = r2.astype(float), n2.astype(float) / N ** 2, lw.astype(float)
        if kind == "counts":
            inp.update(use_counts=1)
            lw = counts[:, 2:7].astype(float) @ np.log(np.arange(2, 7))
    held = {q: torch.from_numpy(v.view(np.int16) if v.dtype == np.uint16 else v).cuda()
            for q, v in dev.items()}
    st = rosen.stats_tensor()
    rosen.rosen_reduce(rosen.rosen_reduce_in(**inp, **{q: v.data_ptr() for q, v in held.items()}),
                       st, rosen.reduce_workspace(C))
    got = rosen.stats_dict(st)
    M = float(lw.max())
    w = np.exp(lw - M)
    ref = {"S0": w, "S1": w * a, "S2": w * b, "Q0": w * w, "Q1_r2": w * w * a, "Q2_r2": w * w * a * a,
           "Q1_rg2": w * w * b, "Q2_rg2": w * w * b * b}
    ref = {q: math.fsum(v) for q, v in ref.items()}
    # (log W up to 18 by counts: its FP64 rounding moves a weight by 2^-49.)
    tol = 4.0 * C * 2.0 ** -53 + 2e-14
    assert got["n"] == got["n_alive"] == C
    assert got["log_max"] == pytest.approx(M, rel=1e-15)
    for q, v in ref.items():
        assert abs(got[q] - v) <= tol * v, (q, got[q], v)
    for x, mean, se, q2 in ((a, "mean_r2", "se_r2", "Q2_r2"), (b, "mean_rg2", "se_rg2", "Q2_rg2")):
        m = ref["S1" if mean == "mean_r2" else "S2"] / ref["S0"]
        v = math.fsum((w * (x - m)) ** 2)
        # The difference of sums loses a factor Q2 / v of the sums' precision.
        assert got[mean] == pytest.approx(m, rel=2 * tol)
        assert got[se] == pytest.approx(math.sqrt(v) / ref["S0"], rel=8 * tol * ref[q2] / v)
