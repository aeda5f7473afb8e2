"""16-bit storage: the step's default kernels are those whose roundings such runs have always had (the
30-column kernel, the line-aligned one on large D3Q19 planes, the row split), bit for bit and in the sums of
the final state, on small and large, walled, driven and periodic lattices. The kernel asked for by name is
the reference: the stored bits must be equal, and so must the FP64 sums, which the same launches form."""
import os

import pytest
import torch

import synth
from paper_2609_09160_gb300 import Solver

pytestmark = pytest.mark.gpu


def _solver(kernel, **kw):
    old = os.environ.pop("LBF_KERNEL", None)
    try:
        if kernel:
            os.environ["LBF_KERNEL"] = kernel
        return Solver(**kw)
    finally:
        os.environ.pop("LBF_KERNEL", None)
        if old is not None:
            os.environ["LBF_KERNEL"] = old


# (lattice, shape, walls, kernel): rows by TMA and loaded directly, below and above 2^20 sites, the wall band of a
# lattice the row split takes, and the sizes from which planes or lattices once changed kernels
CASES = [
    (19, (6, 17, 66), "band", "cta"), (27, (5, 12, 40), "scattered", "cta"), (19, (9, 20, 64), None, "cta"),
    (127, (6, 9, 72), None, "cta"), (27, (70, 130, 128), "band", "cta"), (19, (66, 128, 130), "scattered", "cta"),
    (19, (3, 512, 512), None, "aligned"), (19, (5, 512, 520), "band", "split"), (27, (257, 512, 512), None, "cta"),
]


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_default_kernels_keep_their_roundings(storage, case):
    lattice, shape, walls, kernel = CASES[case]
    mask = None
    if walls == "band":
        mask = synth.channel_walls(shape)
    elif walls == "scattered":
        mask = synth.random_mask(shape, 0.2, seed=41)
    g = torch.Generator(device="cuda").manual_seed(42)
    M0 = torch.empty((10,) + shape, device="cuda").normal_(0.0, 0.01, generator=g)
    M0[0] *= 0.1
    M0[4:] *= 0.1
    kw = dict(shape=shape, lattice=lattice, tau=0.8, storage=storage, force=(1e-6, 0.0, 0.0), mask=mask)
    got = []
    for k in (None, kernel):
        s = _solver(k, **kw)
        s.set_moments(M0)
        s.step(3)
        x = s.new_state()
        s.copy_state(x)
        got.append((s.kernels_per_step, x, s.reduce()))
        del s
    assert got[0][0] == got[1][0]
    assert torch.equal(got[0][1], got[1][1])
    assert list(got[0][2]) == list(got[1][2])
