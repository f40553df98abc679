"""Lattice chains of N >= 160 by the key scan or by bitmap tables: the same chains.

rosen_lattice_grow takes one or the other by length, chain count, restart mode,
interactions and whether conformations are stored; a batch grows members of fewer
chains than the GPU holds by the scan, and a call of at most 32 chains takes the
tables.  Sizes on both sides of each line: N = 208 and 209 (the scan's blocks
shrink), 32 and 33 chains, one and two rounds of resident chains.
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


def grow(rosen, N, C, beta_eps, chain0=0, store=False):
    flags = rosen.ROSEN_STORE_TRACE | rosen.ROSEN_STORE_COORDS if store else 0
    out = rosen.lattice_outputs(N, C, trace=store, coords=store)
    rosen.rosen_lattice_grow(rosen.lattice_params(6, N, C, beta_eps=beta_eps, chain0=chain0,
                                                  flags=flags), out)
    return out


@pytest.mark.parametrize("beta_eps", [0.0, 0.3])
@pytest.mark.parametrize("N", [160, 208, 209])
def test_as_the_class_kernel(rosen, N, beta_eps):
    for C in (1, 32, 33, 5_000, 39_000, 43_000):
        b = rosen.RosenBatch([rosen.ensemble(rosen.ROSEN_MODEL_LATTICE, N, C, 6, 0,
                                             beta_eps=beta_eps)])
        b.run()
        out = grow(rosen, N, C, beta_eps)
        torch.cuda.synchronize()
        for key, v in b.lattice_outputs(0).items():
            assert torch.equal(v, out[key]), (C, key)
        b.close()


@pytest.mark.parametrize("beta_eps", [0.0, 0.3])
@pytest.mark.parametrize("N,C", [(160, 33), (160, 50_001), (185, 55_001), (185, 70_001),
                                 (208, 40_001), (209, 33), (209, 55_001)])
def test_stored_and_not_stored(rosen, N, C, beta_eps):
    out, kept = grow(rosen, N, C, beta_eps), grow(rosen, N, C, beta_eps, store=True)
    torch.cuda.synchronize()
    for key, v in out.items():
        assert torch.equal(v, kept[key]), key
    for chain0 in (0, (C - 32) // 2, C - 32):
        few = grow(rosen, N, 32, beta_eps, chain0, True)
        torch.cuda.synchronize()
        for key, v in few.items():
            whole = kept[key]
            whole = (whole[..., chain0:chain0 + 32] if key in ("trace", "coords")
                     else whole[chain0:chain0 + 32])
            assert torch.equal(v, whole), key


def test_a_stored_chain_that_fills_its_table(rosen):
    # Chain 221724 of seed 3 lies in more blocks than a lane's table holds.
    N, chain0, C = 160, 221_720, 32
    o = oracle.lattice_run(3, N, C, chain0=chain0, trace=True, coords=True)
    block = np.asarray(o["coords"], dtype=np.int64) + 4096 >> 2
    key = np.sort(block[..., 0] + (block[..., 1] << 13) + (block[..., 2] << 26), axis=1)
    assert (1 + (np.diff(key, axis=1) != 0).sum(1)).max() >= 19 * N // 100 + 14
    out = rosen.lattice_outputs(N, C, trace=True, coords=True)
    rosen.rosen_lattice_grow(rosen.lattice_params(3, N, C, chain0=chain0,
                                                  flags=rosen.ROSEN_STORE_TRACE |
                                                  rosen.ROSEN_STORE_COORDS), out)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out["trace"].cpu().numpy().T, o["trace"])
    np.testing.assert_array_equal(out["coords"].permute(2, 0, 1).cpu().numpy(), o["coords"])
