"""Steps with walls against the FP64 oracle on small shapes, by kernels that such lattices reach in other ways too:
the masked 30-column FP32 and FP64 kernel, which large lattices take for scattered walls and for the rows near the
walls of a split step, and 16-bit storage with walls, the default (30-column) and the axis-separated kernel by name.

Tolerances: FP32 and FP64 as everywhere (TOL), relative to the larger of a group's largest value and the scale its
initial values are drawn from. 16-bit storage as for periodic lattices in test_gpu_sep.py: a step stores with one
rounding of at most `unit` of the group's maximum (FP16 2^-10, BF16 2^-7, stochastic rounding moves by up to one
unit), 2 steps add up to at most 4 of them, and one for loading; twenty times that for A, whose maximum is that of
u u; p* is summed from populations of the size of u. Sums: every site's stored value is off by at most that error,
one way or the other, and the sums are those of the stored state: their error is at most its mean times the sites."""
import os

import pytest
import torch

import oracle
import synth
from paper_2609_09160_gb300 import Solver

from _helpers import GROUPS, TOL, as_f32_exact

pytestmark = pytest.mark.gpu
LAT = {19: oracle.D3Q19, 27: oracle.D3Q27}
SCALE = {"p": 1e-3, "u": 0.05, "A": 1e-3}  # synth.random_moments


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


def _mask(kind, shape):
    if kind == "scattered":
        return synth.random_mask(shape, 0.3, seed=72)
    m = synth.channel_walls(shape)
    if kind == "duct":
        m[0], m[-1] = True, True
    return m


@pytest.mark.parametrize("kind", ["band", "scattered", "duct"])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("lattice", [19, 27])
def test_masked_30_column_kernel_matches_oracle(lattice, storage, kind):
    for shape in [(3, 5, 7), (5, 9, 31), (4, 17, 36), (6, 10, 64), (9, 26, 40), (3, 8, 33)]:
        M0, mask = synth.random_moments(shape, seed=71), _mask(kind, shape)
        s = _solver("cta", shape=shape, lattice=lattice, tau=0.7, storage=storage, force=(1e-5, 0.0, -1e-5), mask=mask)
        M1 = M0.clone()
        M1[:, mask] = float("nan")  # solid sites are never read
        s.set_moments(M1.cuda())
        s.step(3)
        want = oracle.lbm.run(LAT[lattice], as_f32_exact(M0) if storage == "f32" else M0, 3, 0.7, force=(1e-5, 0.0, -1e-5), solid=mask)
        got, want = s.moments().cpu()[:, ~mask], want[:, ~mask]
        for g, sl in GROUPS.items():
            assert (got[sl] - want[sl]).abs().max() < TOL[storage] * max(SCALE[g], want[sl].abs().max()), (shape, g)


@pytest.mark.parametrize("kind", ["band", "scattered"])
@pytest.mark.parametrize("kernel", [None, "sep", "sepsmall"])
@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("storage,unit", [("f16", 2.0 ** -10), ("bf16", 2.0 ** -7)])
def test_16_bit_walls_match_oracle(kernel, lattice, storage, unit, kind):
    for rounding in ("stochastic", "nearest"):
        for shape in [(4, 6, 64), (5, 9, 72), (3, 17, 66), (2, 5, 10), (3, 9, 37)]:
            M0, mask = synth.random_moments(shape, seed=74), _mask(kind, shape)
            s = _solver(kernel, shape=shape, lattice=lattice, tau=0.8, storage=storage, rounding=rounding, mask=mask)
            s.set_moments(M0.cuda())
            s.step(2)
            want, got = oracle.lbm.run(LAT[lattice], M0, 2, 0.8, solid=mask)[:, ~mask], s.moments().cpu()[:, ~mask]
            top = {g: want[sl].abs().max().item() for g, sl in GROUPS.items()}
            bound = {"u": 5 * unit * top["u"], "A": 100 * unit * top["A"], "p": 5 * unit * max(top["p"], top["u"])}
            for g, sl in GROUPS.items():
                assert (got[sl] - want[sl]).abs().max().item() < bound[g], (shape, rounding, g)
            sums, n = s.reduce(), got.shape[1]
            assert abs(sums[0] - want[0].sum().item()) < n * bound["p"]
            for k in (1, 2, 3):
                assert abs(sums[k] - want[k].sum().item()) < n * bound["u"], (shape, k)
            assert abs(sums[5] - (want[1:4] ** 2).sum().item()) < n * 2 * bound["u"] * 3 * top["u"]
