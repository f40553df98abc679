"""The reduction at the edges of its tiles and clusters against 64-bit numpy.

A tile is 2048 chains in four quarters of 512 (128 threads, four chains each);
the merge takes 1024 partials a round.  The FP64 sums are compared with numpy's
within 4 n 2^-53 relative (any order of n non-negative terms, weights within
an ulp), whatever lies in an edge: single chains, dead quarters and tiles, the
first chain of a tile alone alive, weights 600 orders of magnitude apart.
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


@pytest.mark.parametrize("C,alive", [
    (1, "all"), (127, "all"), (128, "some"), (129, "all"), (511, "some"), (512, "all"), (513, "first"),
    (2047, "last"), (2048, "some"), (2049, "last"), (4097, "tiles"), (100_001, "some"),
    (1024 * 2048, "some"), (1025 * 2048 + 1, "last"),
])
def test_edges(rosen, C, alive):
    g = np.random.default_rng(C)
    lw = (g.random(C) * 1400 - 700).astype(np.float32)
    if alive == "some":
        lw[g.random(C) < 0.4] = -np.inf
    elif alive == "tiles":
        lw[:2048] = -np.inf
        lw[2048 + 512:4096] = -np.inf
    elif alive != "all":
        keep = 0 if alive == "first" else C - 1
        lw[np.arange(C) != keep] = -np.inf
    r2, rg2 = (g.random(C, dtype=np.float32) * 50 for _ in range(2))
    att = g.integers(1, 9, C).astype(np.uint16)
    dev = [torch.from_numpy(v).cuda() for v in (lw, r2, rg2, att.view(np.int16))]
    inp = rosen.rosen_reduce_in(kind=rosen.ROSEN_REDUCE_OFFLATTICE, N=9, k=7, use_counts=0, C=C,
                                logw=dev[0].data_ptr(), r2_f=dev[1].data_ptr(),
                                rg2_f=dev[2].data_ptr(), attempts=dev[3].data_ptr())
    st = rosen.stats_tensor()
    rosen.rosen_reduce(inp, st, rosen.reduce_workspace(C))
    got = rosen.stats_dict(st)
    live = np.isfinite(lw)
    n = int(live.sum())
    M = float(lw[live].max())
    w, a, b = np.exp(lw[live].astype(np.float64) - M), r2[live].astype(float), rg2[live].astype(float)
    ref = {"S0": w, "S1": w * a, "S2": w * b, "Q0": w * w, "Q1_r2": w * w * a, "Q2_r2": w * w * a * a,
           "Q1_rg2": w * w * b, "Q2_rg2": w * w * b * b}
    ref = {q: math.fsum(v) for q, v in ref.items()}
    tol = 4.0 * n * 2.0 ** -53 + 2e-15
    assert got["n"] == float(att.astype(np.int64).sum()) and got["n_alive"] == n
    assert got["log_max"] == M
    for q, v in ref.items():
        assert abs(got[q] - v) <= tol * v, (q, got[q], v)
    logZ = M + math.log(ref["S0"] / got["n"])
    assert abs(got["logZ"] - logZ) <= tol + 1e-15 * abs(logZ)
    assert abs(got["logZ_norm"] - (logZ - 8 * math.log(7))) <= tol + 2e-15 * (abs(logZ) + 16)
    assert got["mean_r2"] == pytest.approx(ref["S1"] / ref["S0"], rel=2 * tol)
    assert got["mean_rg2"] == pytest.approx(ref["S2"] / ref["S0"], rel=2 * tol)
    assert got["ess"] == pytest.approx(ref["S0"] ** 2 / ref["Q0"], rel=4 * tol)
