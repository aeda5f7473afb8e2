"""The sums of a step over long z-chunks. A thread of the axis-separated kernel makes at most 64 FP32 additions
(of pairs of sites) before its sums go to FP64: it hands them over every 32 planes where it has two rows, and its
chunks end at 64 planes where it has one. Of the additions of equal values half are made in the highest binade,
a quarter in the one below and so on, and each rounds by at most half a unit of its binade, 2^-24 to 2^-25 of the
sum: together at most 64 / 3 * 2^-24 = 1.28e-6 of it (the pairs and the sums across a warp add equal values,
exactly). A uniform flow comes near that; over 96 planes in one FP32 sum it is 2.3e-6 off on D3Q19."""
import os

import pytest
import torch

from paper_2609_09160_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", [19, 27])
def test_sums_over_long_chunks(lattice):
    shape = (96, 8, 64)
    old = {k: os.environ.pop(k, None) for k in ("LBF_KERNEL", "LBF_ZCHUNK")}
    try:
        os.environ.update(LBF_KERNEL="sep", LBF_ZCHUNK="96")
        s = Solver(shape, lattice=lattice, tau=0.8, storage="f32")
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v
    g = torch.Generator().manual_seed(111)
    for u in (0.02 + 0.02 * torch.rand(64, generator=g)).tolist():
        M = torch.zeros((10,) + shape, device="cuda")
        M[0], M[1], M[4] = u / 8, u, u * u
        s.set_moments(M)
        s.step(1)
        sums, now = s.reduce(), s.moments()
        for k, want in ((0, now[0].sum()), (1, now[1].sum()), (5, (now[1:4] ** 2).sum())):
            assert abs(sums[k] / want.item() - 1) < 1.28e-6, (u, k, sums[k], want.item())
