"""A real-space request allocates no more than its outputs, reduction and counters.

A bit per chain is still counted against the budget (what a budget admits does not
change) but not allocated: the server's pool, which keeps what a request returned,
has not grown by it.
"""
import pytest
import torch

from paper_1704_04381_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu
MIB = 1 << 20


@pytest.fixture(scope="module")
def rosen():
    pkg_build.build()
    from paper_1704_04381_gb300 import rosen as r
    r.load()
    return r


def test_counted_but_not_allocated(rosen):
    C = 1 << 29
    used = 13 * C + rosen.rosen_reduce_workspace_size(C)      # 6.6 GiB
    mask = C // 8                                             # 64 MiB
    req = rosen.request(rosen.ROSEN_MODEL_OFFLATTICE, 2, C, 3, 0, k=1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    srv = rosen.RosenServer(mem_budget_bytes=used + mask + MIB)
    try:
        st, res = srv.wait(srv.submit(req), 60)
        assert st == rosen.ROSEN_OK and res["status"] == rosen.ROSEN_OK, res
        assert res["stats"]["n"] == C
        assert free - torch.cuda.mem_get_info()[0] < used + mask * 3 // 4
        assert srv.info()["bytes_in_use"] == 0
    finally:
        srv.close()
    srv = rosen.RosenServer(mem_budget_bytes=used + mask // 2)
    try:
        with pytest.raises(rosen.RosenError):
            srv.submit(req)
    finally:
        srv.close()
