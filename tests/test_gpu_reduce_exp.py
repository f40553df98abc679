"""The weights' exponential of the reduction against a longer format.

Of two chains with log W = 0 and log W = x < 0, R_ee^2 = 0 and 1, the sum S1 is
exactly the weight exp(x): its error can be read off.  It is no larger than that
of CUDA's double exp (documented: at most 1 ulp, measured 0.86): the rounding of
the last sum is half an ulp, the polynomial, the argument and the table's second
word add some hundredths.
"""
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


@pytest.mark.parametrize("low", [1e-3, 1.0, 30.0, 700.0])
def test_weight_within_its_rounding(rosen, low):
    n = 1500
    x = -(np.random.default_rng(int(low)).random(n) * low).astype(np.float32)
    x[0] = -low
    lw = torch.zeros(n, 2)
    lw[:, 1] = torch.from_numpy(x)
    lw = lw.cuda()
    r2 = torch.tensor([0.0, 1.0]).cuda()
    st = torch.zeros(n, len(rosen.STAT_KEYS), dtype=torch.float64, device="cuda")
    ws = rosen.reduce_workspace(2)
    for q in range(n):
        inp = rosen.rosen_reduce_in(kind=rosen.ROSEN_REDUCE_OFFLATTICE, N=4, k=3, use_counts=0, C=2,
                                    logw=lw[q].data_ptr(), r2_f=r2.data_ptr(), rg2_f=r2.data_ptr())
        rosen.rosen_reduce(inp, st[q], ws)
    got = st[:, list(rosen.STAT_KEYS).index("S1")].cpu().numpy()
    ref = np.exp(x.astype(np.longdouble))
    err = np.abs((got.astype(np.longdouble) - ref) / np.spacing(got).astype(np.longdouble))
    assert float(err.max()) < 0.56, float(err.max())
    assert float(err.mean()) < 0.26, float(err.mean())
