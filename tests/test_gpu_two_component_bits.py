"""Two components: the values of a run do not depend on how its launches are cut. Where grad phi is small its
direction hangs on the last bits of phi and u, so a change of rounding anywhere reaches the interface: the step's
default kernel is the 30-column one, bit for bit, and the phase field of a lattice that is filled with copies of a few
planes advances as that of those planes does, wherever the phase-field kernels' z-chunks begin. By name the axis-separated kernel agrees with the oracle."""
import os

import pytest
import torch

import oracle
import synth
from paper_2609_09160_gb300 import Solver

from _helpers import GROUPS, TOL, as_f32_exact

pytestmark = pytest.mark.gpu
EQUAL = dict(rho_l=1.0, rho_h=1.0, tau_l=0.8, tau_h=0.8, sigma=0.01, width=4.0, diffusivity=0.1)
CONTRAST = dict(EQUAL, rho_l=0.6, rho_h=1.4, tau_h=1.1, body_accel=(1e-6, 0.0, 2e-6))


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


def _start(shape, storage):
    M0 = synth.random_moments(shape, seed=131)
    phi0 = (0.5 + 0.4 * synth.random_field(shape, 0.5, seed=132)[0]).clamp(0, 1)
    dt = torch.float64 if storage == "f64" else torch.float32
    return M0.to("cuda", dt), phi0.to("cuda", dt)


@pytest.mark.parametrize("two", [EQUAL, CONTRAST])
@pytest.mark.parametrize("walls", [False, True])
def test_default_kernel_keeps_its_values(two, walls):
    for shape in [(9, 26, 64), (5, 17, 37), (40, 128, 256)]:
        mask = synth.random_mask(shape, 0.15, seed=133) if walls else None
        got = []
        for kernel in (None, "cta"):
            s = _solver(kernel, shape=shape, lattice=19, storage="f32", two_component=two, mask=mask)
            s.set_moments(*_start(shape, "f32"))
            s.step(4)
            x = s.new_state()
            s.copy_state(x)
            got.append((x, s.phi(), s.reduce()))
        assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1]) and list(got[0][2]) == list(got[1][2])


@pytest.mark.parametrize("two", [EQUAL, CONTRAST])
@pytest.mark.parametrize("storage,lattice", [("f32", 19), ("f64", 19), ("f32", 27)])
def test_phase_field_does_not_depend_on_chunks(storage, lattice, two):
    part = (10, 20, 37)
    M0, phi0 = _start(part, storage)
    got = []
    for n in (1, 7):
        s = Solver((part[0] * n,) + part[1:], lattice=lattice, storage=storage, two_component=two)
        s.set_moments(M0.repeat(1, n, 1, 1), phi0.repeat(n, 1, 1))
        s.step(1)
        got.append(s.phi())
    assert torch.equal(got[1], got[0].repeat(7, 1, 1))


@pytest.mark.parametrize("contrast", [False, True])
@pytest.mark.parametrize("walls", [False, True])
def test_axis_separated_kernel_matches_oracle(contrast, walls):
    """As test_sep_two_components_match_oracle in test_gpu_sep.py, whose default is another kernel now."""
    for shape in [(3, 5, 7), (4, 6, 64), (5, 9, 68), (3, 17, 67), (9, 13, 132)]:
        M0 = synth.random_moments(shape, seed=80)
        phi0 = as_f32_exact((0.5 + 0.4 * synth.random_field(shape, 0.5, seed=81)[0]).clamp(0, 1))
        mask = synth.random_mask(shape, 0.15, seed=82) if walls else None
        two = dict(CONTRAST if contrast else EQUAL, body_accel=(1e-6, 0.0, 2e-6))
        s = _solver("sep", shape=shape, lattice=19, storage="f32", two_component=two, mask=mask, force=(1e-6, -1e-6, 0.0))
        s.set_moments(M0.cuda(), phi0.cuda())
        s.step(3)
        want, wphi = oracle.phase.run(oracle.D3Q19, as_f32_exact(M0), phi0, 3, two["tau_l"], two["tau_h"], 0.01, 4.0, 0.1, rho_l=two["rho_l"],
                                      rho_h=two["rho_h"], body=(1e-6, -1e-6, 0.0), solid=mask, body_accel=(1e-6, 0.0, 2e-6))
        for g, sl in GROUPS.items():
            scale = max({"p": 1e-3, "u": 0.05, "A": 1e-3}[g], want[sl].abs().max().item())
            assert (s.moments().cpu()[sl] - want[sl]).abs().max().item() < TOL["f32"] * scale, (shape, g)
        assert (s.phi().cpu() - wphi).abs().max() < TOL["f32"] * wphi.abs().max(), shape
