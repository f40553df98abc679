"""Reductions of few chains: one merging block, quarters of a tile without chains.

Up to 128 tiles one block merges the partials, beyond them a cluster of eight;
blocks of a short tile's empty quarters add nothing.  The statistics do not
depend on which: an ensemble reduced alone (one block) equals, bit for bit, the
same ensemble in a batch whose largest member makes the batch use clusters, and
in one of small members only.
"""
import pytest
import torch

from paper_1704_04381_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu
SIZES = (1, 127, 512, 513, 1024, 1025, 2047, 2048, 2049, 2048 + 512, 2048 + 513, 100_001, 128 * 2048)


@pytest.fixture(scope="module")
def rosen():
    pkg_build.build()
    from paper_1704_04381_gb300 import rosen as r
    r.load()
    return r


@pytest.mark.parametrize("largest", [0, 128 * 2048 + 1])
def test_alone_and_in_a_batch(rosen, largest):
    sizes = SIZES + ((largest,) if largest else ())
    ens = [rosen.ensemble(rosen.ROSEN_MODEL_LATTICE, 24, C, 7, e, beta_eps=0.3 * (e % 2))
           for e, C in enumerate(sizes)]
    b = rosen.RosenBatch(ens)
    b.run()
    got = b.stats()
    torch.cuda.synchronize()
    for e, x in enumerate(ens):
        out = rosen.lattice_outputs(x.N, x.C)
        rosen.rosen_lattice_grow(rosen.lattice_params(7, x.N, x.C, ensemble=e, beta_eps=x.beta_eps),
                                 out)
        st = rosen.stats_tensor()
        rosen.rosen_reduce(rosen.lattice_reduce_in(out, x.N, int(x.beta_eps == 0.0)), st,
                           rosen.reduce_workspace(x.C))
        torch.cuda.synchronize()
        assert torch.equal(got[e].view(torch.int64), st.view(torch.int64)), (e, x.C)
    b.close()
