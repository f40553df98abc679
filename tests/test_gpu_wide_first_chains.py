"""A warp's first hard-sphere chains on shared memory another kernel left full.

offlattice_wide_kernel clears a chain's shared memory and then marks its beads
as not placed, the same words from other lanes of the group.  The first chains
of every group shape are compared bit for bit with those of the long-chain
kernel, which keeps its chains in device memory, each time after Lennard-Jones
chains have filled the shared memory of every SM.
"""
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


@pytest.mark.parametrize("N,k,C", [(5, 16, 1), (33, 32, 5), (64, 32, 600), (130, 32, 40_000),
                                   (300, 64, 9_001), (1024, 32, 300)])
def test_first_chains(rosen, N, k, C):
    full = rosen.offlattice_outputs(512, 2_000)
    fill = rosen.offlattice_params(1, 512, 2_000, 8, potential=rosen.ROSEN_LJ, beta_eps=0.1)
    out = [rosen.offlattice_outputs(N, C, trace=True, coords=True, counters=True) for _ in range(2)]
    p = rosen.offlattice_params(8, N, C, k, lanes_per_chain=32,
                                flags=rosen.ROSEN_STORE_TRACE | rosen.ROSEN_STORE_COORDS)
    rosen.rosen_offlattice_grow_long(p, out[0], rosen.offlattice_long_workspace(N, C))
    for _ in range(4):
        for v in out[1].values():
            v.zero_()
        rosen.rosen_offlattice_grow(fill, full)
        rosen.rosen_offlattice_grow(p, out[1])
        torch.cuda.synchronize()
        for key in out[0]:
            assert torch.equal(*(o[key].view(torch.uint8) for o in out)), key
