"""Batch members that their own kernel grows faster than the class kernel.

Hard spheres and lattice chains of N >= 160 have faster kernels for one ensemble
than the class kernels of a batch: members that fill the GPU once get them, as
those that filled it four times with the earlier kernels did (hard spheres, N =
64: 38912 chains; lattice, N = 512: 58368).  Their outputs are those of the
single-ensemble calls, bit for bit, and so are the smaller members'.
"""
import json

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


def test_members_that_fill_the_gpu_get_their_own_launch(rosen):
    L, R = rosen.ROSEN_MODEL_LATTICE, rosen.ROSEN_MODEL_OFFLATTICE
    ens = [rosen.ensemble(R, 64, 38_912, 1, 0, k=32), rosen.ensemble(R, 60, 3_000, 1, 1, k=32),
           rosen.ensemble(L, 512, 58_368, 1, 2), rosen.ensemble(L, 500, 900, 1, 3, beta_eps=0.2),
           rosen.ensemble(R, 40, 3_000, 1, 4, k=32, potential=rosen.ROSEN_LJ, beta_eps=0.3)]
    b = rosen.RosenBatch(ens)
    b.tune()
    b.run()
    own, lanes = {}, {}
    for c in json.loads(b.describe()):
        own.update(zip(c["members"], c["own_launch"]))
        lanes.update(zip(c["members"], c["member_lanes"]))
    assert [own[e] for e in range(5)] == [1, 0, 1, 0, 0]
    for e, x in enumerate(ens):
        if x.model == L:
            out = rosen.lattice_outputs(x.N, x.C)
            rosen.rosen_lattice_grow(rosen.lattice_params(1, x.N, x.C, ensemble=e,
                                                          beta_eps=x.beta_eps), out)
            mine = b.lattice_outputs(e)
        else:
            out = rosen.offlattice_outputs(x.N, x.C)
            rosen.rosen_offlattice_grow(
                rosen.offlattice_params(1, x.N, x.C, x.k, ensemble=e, potential=x.potential,
                                        beta_eps=x.beta_eps, lanes_per_chain=lanes[e]), out)
            mine = b.offlattice_outputs(e)
        torch.cuda.synchronize()
        for key, v in mine.items():
            assert torch.equal(v, out[key]), (e, key)
    b.close()
