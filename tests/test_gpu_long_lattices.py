"""Lattices that are very long in y or z: a grid holds at most 65535 blocks along each, and the step's tiles and
z-chunks differ in height. Every lattice that the 30-column kernel can take is stepped, and agrees with the FP64
oracle at the tolerances of the other tests (TOL), relative to the scale the values are drawn from."""
import pytest
import torch

import oracle
import synth
from paper_2609_09160_gb300 import Solver

from _helpers import GROUPS, TOL, as_f32_exact

pytestmark = pytest.mark.gpu
LAT = {19: oracle.D3Q19, 27: oracle.D3Q27, 127: oracle.D3Q27H}
SCALE = {"p": 1e-3, "u": 0.05, "A": 1e-3}  # synth.random_moments


def _check(got, want, tol):
    for g, sl in GROUPS.items():
        assert (got[sl].cpu() - want[sl]).abs().max().item() < tol * max(SCALE[g], want[sl].abs().max().item()), g


# (nz, ny, nx): one block more than 65535 tiles of 2 rows (FP64), of 4 rows (the short FP32 tile)
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("lattice,storage,shape", [(19, "f64", (1, 131074, 4)), (27, "f64", (1, 131074, 3)),
                                                   (19, "f32", (1, 262146, 3)), (19, "f64", (1, 131070, 4))])
def test_many_rows(lattice, storage, shape, walls):
    M0 = synth.random_moments(shape, seed=91)
    mask = synth.random_mask(shape, 0.1, seed=92) if walls else None
    s = Solver(shape, lattice=lattice, tau=0.8, storage=storage, mask=mask)
    s.set_moments(M0.cuda())
    s.step(2)
    s.synchronize()
    want = oracle.lbm.run(LAT[lattice], as_f32_exact(M0) if storage == "f32" else M0, 2, 0.8, solid=mask)
    _check(s.moments(), want, TOL[storage])


# one block more than 65535 chunks of the phase field's 6 planes. No diffusivity: the interface flux, whose direction
# grad phi / |grad phi| is as ill conditioned as the gradient is small somewhere among 1.5 million sites (two orders
# of summation differ by 1e-9 in FP64), then has no weight
@pytest.mark.parametrize("contrast", [False, True])
@pytest.mark.parametrize("storage", ["f32", "f64"])
def test_many_planes_two_components(storage, contrast):
    shape = (393216, 2, 2)
    M0 = synth.random_moments(shape, seed=93)
    phi0 = as_f32_exact((0.5 + 0.4 * synth.random_field(shape, 0.5, seed=94)[0]).clamp(0, 1))
    kw = dict(rho_l=0.7 if contrast else 1.0, rho_h=1.3 if contrast else 1.0)
    two = dict(tau_l=0.8, tau_h=1.1, sigma=0.01, width=4.0, diffusivity=0.0, **kw)
    s = Solver(shape, lattice=19, storage=storage, two_component=two)
    s.set_moments(M0.cuda(), phi0.cuda())
    s.step(2)
    s.synchronize()
    want, wphi = oracle.phase.run(oracle.D3Q19, as_f32_exact(M0) if storage == "f32" else M0, phi0, 2, 0.8, 1.1, 0.01, 4.0, 0.0, **kw)
    _check(s.moments(), want, TOL[storage])
    assert (s.phi().cpu() - wphi).abs().max() < TOL[storage]
