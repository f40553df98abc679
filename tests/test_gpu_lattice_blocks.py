"""Parity of the bitmap-table lattice kernel (mid-length chains) with the oracle.

Bit-exact per chain, at the first length that takes it and the longest, with
ragged counts, restart mode, traces on (the lanes of a warp stay in step) and
off (they do not), and chains that fill their lane's table (found by their
number of 4x4x4 blocks) and are grown again with the whole warp's.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1704_04381_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosen():
    pkg_build.build()
    from paper_1704_04381_gb300 import rosen as r
    r.load()
    return r


def grow(rosen, N, C, beta_eps, chain0, attempts, store):
    flags = rosen.ROSEN_STORE_TRACE | rosen.ROSEN_STORE_COORDS if store else 0
    out = rosen.lattice_outputs(N, C, trace=store, coords=store, attempts=True)
    rosen.rosen_lattice_grow(rosen.lattice_params(3, N, C, beta_eps=beta_eps, chain0=chain0,
                                                  flags=flags, max_attempts=attempts), out)
    torch.cuda.synchronize()
    return {k: v.cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("N,C,beta_eps,chain0,fills", [
    (160, 700, 0.0, 0, False), (160, 33, 0.0, 221_720, True), (160, 64, 0.0, 568_100, True),
    (161, 500, 0.3, 9, False), (256, 33, 0.0, 25_560, False),
    (256, 1, 0.6, 4, False), (512, 300, 0.0, 0, False), (512, 300, 0.4, 1, False),
])
def test_matches_the_oracle(rosen, N, C, beta_eps, chain0, fills):
    o = oracle.lattice_run(3, N, C, beta_eps=beta_eps, chain0=chain0, trace=True, coords=True)
    if fills:
        block = np.asarray(o["coords"], dtype=np.int64) + 4096 >> 2
        key = np.sort(block[..., 0] + (block[..., 1] << 13) + (block[..., 2] << 26), axis=1)
        assert (1 + (np.diff(key, axis=1) != 0).sum(1)).max() >= 19 * N // 100 + 14
    g = grow(rosen, N, C, beta_eps, chain0, 0, True)
    np.testing.assert_array_equal(g["trace"].T, o["trace"])
    np.testing.assert_array_equal(np.transpose(g["coords"], (2, 0, 1)), o["coords"])
    np.testing.assert_array_equal(g["counts"].view(np.uint16), o["counts"])
    np.testing.assert_array_equal(g["r2"], o["r2"])
    np.testing.assert_array_equal(g["n2rg2"], o["n2rg2"])
    plain = grow(rosen, N, C, beta_eps, chain0, 0, False)
    for key in plain:
        np.testing.assert_array_equal(plain[key], g[key], err_msg=key)


@pytest.mark.parametrize("N,beta_eps,store", [(160, 0.0, False), (300, 0.4, True), (512, 0.0, True)])
def test_restart_mode(rosen, N, beta_eps, store):
    C, cap = 400, 40
    o = oracle.lattice_run(3, N, C, beta_eps=beta_eps, max_attempts=cap, trace=store, coords=store)
    g = grow(rosen, N, C, beta_eps, 0, cap, store)
    np.testing.assert_array_equal(g["attempts"].view(np.uint16), o["attempts"])
    assert (o["attempts"] > 1).any()
    np.testing.assert_array_equal(g["counts"].view(np.uint16), o["counts"])
    np.testing.assert_array_equal(g["r2"], o["r2"])
    np.testing.assert_array_equal(g["n2rg2"], o["n2rg2"])
