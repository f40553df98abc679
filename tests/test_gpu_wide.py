"""Hard spheres by the few-lanes kernel against the long-chain kernel.

rosen_offlattice_grow and rosen_offlattice_grow_long grow hard spheres with
different device code (few lanes per chain and a scan; 16 or 32 lanes and a
cell grid) but the same arithmetic, so every output, the FP64 re-decision
count and the listed-bead count included, is equal bit for bit.  The sizes
are the edges of the kernel's shapes: lanes per chain, trials per lane (k),
scan blocks and scan words (N), and few chains (wider groups).
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


@pytest.mark.parametrize("N,k,C,lanes,sigma,attempts", [
    (2, 1, 9, 16, 1.0, 0), (3, 8, 1, 16, 1.0, 0), (16, 9, 7, 16, 1.0, 0), (17, 16, 5001, 16, 1.0, 0),
    (64, 24, 12_001, 16, 1.0, 0), (64, 32, 20_003, 16, 1.0, 0), (65, 33, 9_001, 32, 1.0, 0),
    (66, 64, 7_001, 16, 1.0, 0), (30, 65, 6_001, 32, 1.0, 0), (31, 128, 6_001, 32, 1.0, 0),
    (128, 32, 20_003, 32, 1.0, 0), (129, 32, 9_001, 32, 1.0, 0), (256, 32, 2_001, 16, 1.0, 0),
    (257, 48, 301, 32, 1.0, 0), (512, 32, 301, 32, 1.0, 0), (513, 100, 65, 32, 1.0, 0),
    (1024, 16, 33, 16, 1.0, 0), (40, 16, 20_003, 16, 1.5, 0), (40, 16, 3_001, 16, 1.5, 7),
    (50, 8, 12_001, 16, 1.6, 40), (30, 16, 3_001, 16, 0.0, 0), (30, 16, 3_001, 16, 0.3, 0),
])
def test_same_chains_as_the_long_kernel(rosen, N, k, C, lanes, sigma, attempts):
    outs = []
    for long in (False, True):
        out = rosen.offlattice_outputs(N, C, trace=True, coords=True, counters=True, attempts=True)
        p = rosen.offlattice_params(21, N, C, k, sigma=sigma, chain0=5, ensemble=2,
                                    flags=rosen.ROSEN_STORE_TRACE | rosen.ROSEN_STORE_COORDS,
                                    lanes_per_chain=lanes, max_attempts=attempts)
        if long:
            rosen.rosen_offlattice_grow_long(p, out, rosen.offlattice_long_workspace(N, C))
        else:
            rosen.rosen_offlattice_grow(p, out)
        outs.append(out)
    torch.cuda.synchronize()
    for key in outs[0]:
        a, b = (o[key].view(torch.uint8) for o in outs)
        assert torch.equal(a, b), key
