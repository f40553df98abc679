"""The hard-sphere kernel's fast trial directions against the ones it commits.

A step that the fast directions decide must be one that dir32's decide, and
alike: the kernel widens its band by kFastDir |g| (kFastDir bounds the Euclidean
norm of the difference of twice the two directions) and by the roundings of two
sums of three products.  The norm is at most the sum of its part in the angle
(every one of the 2^24, at s = 1, where products with s are exact), its part in s
(every polar word, at angle 0) and the rounding of both sides' products with s
(components of 2u below 2: half an ulp is 2^-24, two components, two sides).
"""
import os
import re

import numpy as np
import pytest
import torch

from paper_1704_04381_gb300 import build as pkg_build

pytestmark = pytest.mark.gpu
PRODUCTS = 2 * 2.0 ** 0.5 * 2.0 ** -24


@pytest.fixture(scope="module")
def rosen():
    pkg_build.build()
    from paper_1704_04381_gb300 import rosen as r
    r.load()
    return r


@pytest.fixture(scope="module")
def bound():
    with open(os.path.join(pkg_build.CSRC, "offlattice_wide.cuh")) as f:
        return float(re.search(r"kFastDir = ([0-9.e+-]+);", f.read()).group(1))


def norms(rosen, a, b):
    """|2u fast - 2u| of every pair of words; z must agree exactly."""
    words = torch.stack([a, b], 1).to(torch.int32).contiguous()     # (the low 32 bits)
    u, v = (torch.empty(len(a), 3, dtype=torch.float32, device="cuda") for _ in range(2))
    rosen.rosen_sphere_points(words, u)
    rosen.rosen_sphere_points_fast(words, v)
    assert torch.equal(u[:, 2], v[:, 2])
    return 2.0 * float((u.double() - v.double()).square().sum(1).max().sqrt())


def words24():
    w = torch.arange(1 << 24, device="cuda", dtype=torch.int64) << 8
    return torch.where(w >= 1 << 31, w - (1 << 32), w)


def test_all_angles_and_all_polar_words(rosen, bound):
    w = words24()
    angle = norms(rosen, torch.full_like(w, -(1 << 31)), w)
    polar = norms(rosen, w, torch.zeros_like(w))
    assert angle + polar + PRODUCTS < bound, (angle, polar)


def test_random_directions(rosen, bound):
    g = torch.Generator("cuda").manual_seed(5)
    for _ in range(8):
        a, b = (torch.randint(-(1 << 31), 1 << 31, (1 << 24,), generator=g, device="cuda")
                for _ in range(2))
        assert norms(rosen, a, b) < bound


def test_every_chain_as_off_chain_in_number_of_decisions(rosen):
    # 2 10^5 chains meet about 4000 steps within the bands: the re-decided ones
    # and the paths are those of the long-chain kernel.
    N, k, C = 64, 32, 200_000
    outs = [rosen.offlattice_outputs(N, C, trace=True, counters=True) for _ in range(2)]
    p = rosen.offlattice_params(77, N, C, k, lanes_per_chain=16, flags=rosen.ROSEN_STORE_TRACE)
    rosen.rosen_offlattice_grow(p, outs[0])
    rosen.rosen_offlattice_grow_long(p, outs[1], rosen.offlattice_long_workspace(N, C))
    torch.cuda.synchronize()
    assert int(outs[0]["counters"][0]) > 2_000
    for key in outs[0]:
        assert torch.equal(*(o[key].view(torch.uint8) for o in outs)), key
