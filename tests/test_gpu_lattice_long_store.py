"""Stored long athermal chains: the rows after a dead end, lanes that start together.

The rows a trapped chain leaves are written by its whole warp, and the lanes of a
warp take their next chains together.  With many dead ends and few tables (ragged
warps, several chains per lane) every chain is the oracle's, and stored and not
stored calls agree.
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


@pytest.mark.parametrize("N,C,tables,attempts,flags", [
    (700, 75, 75, 0, 3), (1500, 130, 33, 0, 3), (1500, 40, 1, 0, 1), (1200, 97, 50, 3, 2),
    (2, 70, 3, 0, 3),
])
def test_rows_and_chains(rosen, N, C, tables, attempts, flags):
    per = rosen.rosen_lattice_long_workspace_size(N, 2) - rosen.rosen_lattice_long_workspace_size(N, 1)
    head = rosen.rosen_lattice_long_workspace_size(N, 1) - per
    ws = torch.empty((head + tables * per) // 8, dtype=torch.int64, device="cuda")
    out = rosen.lattice_outputs(N, C, trace=flags & 1 > 0, coords=flags & 2 > 0, attempts=True)
    plain = rosen.lattice_outputs(N, C, attempts=True)
    for o, f in ((out, flags), (plain, 0)):
        for v in o.values():
            v.fill_(85)
        rosen.rosen_lattice_grow_long(rosen.lattice_params(9, N, C, flags=f, max_attempts=attempts), o,
                                      ws)
    torch.cuda.synchronize()
    for key, v in plain.items():
        assert torch.equal(v, out[key]), key
    o = oracle.lattice_run(9, N, C, max_attempts=max(attempts, 1), trace=True, coords=True)
    np.testing.assert_array_equal(out["counts"].cpu().numpy().view(np.uint16), o["counts"])
    assert N < 700 or attempts or (o["counts"][:, 0] > 0).sum() > 5
    if flags & 1:
        np.testing.assert_array_equal(out["trace"].cpu().numpy().T, o["trace"])
    if flags & 2:
        np.testing.assert_array_equal(out["coords"].permute(2, 0, 1).cpu().numpy(), o["coords"])
