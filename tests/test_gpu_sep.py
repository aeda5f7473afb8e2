"""The axis-separated fused kernel (both tiles: LBF_KERNEL=sep, sepsmall; rows by TMA and by cp.async)
against the FP64 oracle, on shapes at the edges of its tiles: rows shorter than, equal to and just
longer than one tile, a last tile moved left, odd rows, partial row groups, more rows than one tile,
one plane, chunk seams; walls at tile seams and scattered, force fields, the 16-bit codecs; and the
row split's cyclic row range.

Tolerances: FP32/FP64 as everywhere (TOL), relative to the larger of a group's largest value and the
scale its initial values are drawn from (a lattice of a few sites may draw small ones only, and p* is
summed from populations of the size of u). 16-bit storage: a step stores with one rounding of relative
size at most 2^-10 (FP16) or 2^-7 (BF16, stochastic rounding moves by up to one unit) of the stored
value, which is at most the group's maximum; after n steps the errors add to at most 2 n of them (the
collision at most about doubles N), plus one for loading."""
import os

import pytest
import torch

import oracle
import synth
from paper_2609_09160_gb300 import Solver

from _helpers import GROUPS, TOL, as_f32_exact, group_errors

pytestmark = pytest.mark.gpu
LAT = {19: oracle.D3Q19, 27: oracle.D3Q27, 127: oracle.D3Q27H}
STEPS = 3


SCALE = {"p": 1e-3, "u": 0.05, "A": 1e-3}  # synth.random_moments


def _errors(got, want):
    err = group_errors(got, want)
    for g, sl in GROUPS.items():
        top = want[sl].abs().max().item()
        err[g] *= top / max(top, SCALE[g])
    return err


def _solver(kernel, zchunk=None, **kw):
    old = {k: os.environ.pop(k, None) for k in ("LBF_KERNEL", "LBF_ZCHUNK")}
    try:
        if kernel:
            os.environ["LBF_KERNEL"] = kernel
        if zchunk:
            os.environ["LBF_ZCHUNK"] = str(zchunk)
        return Solver(**kw)
    finally:
        for k, v in old.items():
            os.environ.pop(k, None)
            if v is not None:
                os.environ[k] = v


# (nz, ny, nx): one site; fewer columns than a tile; exactly one tile; one tile and 4 more (TMA, moved
# tile); odd rows; two and a bit tiles of rows
SHAPES = [(1, 1, 1), (3, 5, 7), (4, 6, 64), (5, 9, 68), (3, 17, 67), (7, 12, 132), (2, 33, 40)]


@pytest.mark.parametrize("kernel", ["sep", "sepsmall"])
@pytest.mark.parametrize("storage", ["f32", "f64"])
@pytest.mark.parametrize("lattice", [19, 27, 127])
def test_sep_periodic_matches_oracle(kernel, storage, lattice):
    for shape in SHAPES:
        M0 = synth.random_moments(shape, seed=70)
        kw = dict(force=(2e-5, -1e-5, 3e-5))
        for z in (None, 2):
            s = _solver(kernel, z, shape=shape, lattice=lattice, tau=0.8, storage=storage, **kw)
            s.set_moments(M0.cuda())
            s.step(STEPS)
            want = oracle.lbm.run(LAT[lattice], as_f32_exact(M0) if storage == "f32" else M0, STEPS, 0.8, **kw)
            err = _errors(s.moments(), want)
            assert max(err.values()) < TOL[storage], (shape, z, err)
            ref = oracle.diagnostics.reductions(want, None)
            got = s.reduce()
            mag = [want[0].abs().sum()] + [want[1 + i].abs().sum() for i in range(3)] + [1.0, (want[1:4] ** 2).sum()]
            for k in (0, 1, 2, 3):
                assert abs(got[k] - float(ref[k])) <= 10 * TOL[storage] * float(mag[k]), (shape, k)


@pytest.mark.parametrize("kernel", ["sep", "sepsmall"])
@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("kind", ["band", "scattered", "field", "wall_x"])
def test_sep_walls_and_fields_match_oracle(kernel, lattice, kind):
    for storage in ("f32", "f64"):
        for shape in SHAPES[1:]:
            M0 = synth.random_moments(shape, seed=71)
            mask = field = None
            if kind == "band":
                mask = synth.channel_walls(shape)
            elif kind == "scattered":
                mask = synth.random_mask(shape, 0.3, seed=72)
            elif kind == "wall_x":
                mask = torch.zeros(shape, dtype=torch.bool)
                mask[..., 0] = mask[..., -1] = True
            if kind in ("field", "wall_x"):
                field = synth.random_field(shape, 1e-4, seed=73)
            cdt = torch.float32 if storage == "f32" else torch.float64
            exact = (lambda t: as_f32_exact(t)) if storage == "f32" else (lambda t: t)
            s = _solver(kernel, 2, shape=shape, lattice=lattice, tau=0.7, storage=storage, force=(1e-5, 0.0, -1e-5), mask=mask,
                        force_field=None if field is None else field.to("cuda", cdt))
            M1 = M0.clone()
            if mask is not None:
                M1[:, mask] = float("nan")  # solid sites are never read
            s.set_moments(M1.cuda())
            s.step(STEPS)
            F = torch.tensor([1e-5, 0.0, -1e-5], dtype=torch.float64).reshape(3, 1, 1, 1).expand((3,) + shape)
            want = oracle.lbm.run(LAT[lattice], exact(M0), STEPS, 0.7, force=F if field is None else F + exact(field), solid=mask)
            fluid = slice(None) if mask is None else ~mask
            err = _errors(s.moments().cpu()[:, fluid], want[:, fluid])
            assert max(err.values()) < TOL[storage], (shape, storage, err)


@pytest.mark.parametrize("kernel", ["sep", "sepsmall"])
@pytest.mark.parametrize("lattice", [19, 27, 127])
@pytest.mark.parametrize("storage,unit", [("f16", 2.0 ** -10), ("bf16", 2.0 ** -7)])
def test_sep_16bit_matches_oracle(kernel, lattice, storage, unit):
    for rounding in ("stochastic", "nearest"):
        for shape in [(4, 6, 64), (5, 9, 72), (3, 17, 66), (2, 5, 10)]:
            M0 = synth.random_moments(shape, seed=74)
            s = _solver(kernel, 2, shape=shape, lattice=lattice, tau=0.8, storage=storage, rounding=rounding)
            s.set_moments(M0.cuda())
            s.step(2)
            want = oracle.lbm.run(LAT[lattice], M0, 2, 0.8)
            err = group_errors(s.moments(), want)
            # p* is summed from populations of the size of u: its error follows the u group
            scale = (want[1:4].abs().max() / want[0].abs().max()).item()
            assert err["u"] < 5 * unit and err["A"] < 5 * unit * 20 and err["p"] < 5 * unit * max(1.0, scale), (shape, err)


@pytest.mark.parametrize("walls", [(0, -1), (60,), (125, 126)])
def test_sep_row_split_matches_masked_kernel(walls):
    """Walls in a band of rows of a lattice large enough for the split: the clean rows, a cyclic range that
    may pass y = ny - 1, run the axis-separated kernel. Compared with the single masked 30-column launch
    at twice the FP32 tolerance (each is within it of the oracle), sums included."""
    shape = (34, 130, 260)
    mask = torch.zeros(shape, dtype=torch.bool)
    for y in walls:
        mask[:, y] = True
    M0 = synth.random_moments(shape, seed=75)
    for field in (None, synth.random_field(shape, 1e-4, seed=76).to("cuda", torch.float32)):
        kw = dict(shape=shape, lattice=19, tau=0.7, storage="f32", force=(1e-5, -2e-6, 3e-6), mask=mask, force_field=field)
        a, b = _solver(None, **kw), _solver("cta", **kw)
        assert a.kernels_per_step == 2 and b.kernels_per_step == 1
        for s in (a, b):
            s.set_moments(M0.cuda())
            s.step(4)
        assert max(group_errors(a.moments(), b.moments()).values()) < 2 * TOL["f32"]
        ra, rb = a.reduce(), b.reduce()
        mag = [M0[0].abs().sum().item()] + [M0[1 + i].abs().sum().item() for i in range(3)] + [1.0, (M0[1:4] ** 2).sum().item()]
        for k in (0, 1, 2, 3, 5):
            assert abs(ra[k] - rb[k]) <= 2 * TOL["f32"] * mag[k], (k, ra[k], rb[k])
        # a step between caller buffers gives the same bits as the context's own step
        x = a.new_state()
        a.copy_state(x)
        y = x.clone()
        a.step_state(x, y)
        a.step(1)
        a.copy_state(x)
        assert torch.equal(x, y)


@pytest.mark.parametrize("contrast", [False, True])
@pytest.mark.parametrize("walls", [False, True])
def test_sep_two_components_match_oracle(contrast, walls):
    """Two components on D3Q19 FP32 (the axis-separated kernel, the default there) at the edges of its
    tiles, moments and phase field against the oracle; rows by TMA (nx 64, 68, 132) and cp.async."""
    for shape in [(3, 5, 7), (4, 6, 64), (5, 9, 68), (3, 17, 67), (9, 13, 132)]:
        M0 = synth.random_moments(shape, seed=80)
        phi0 = as_f32_exact((0.5 + 0.4 * synth.random_field(shape, 0.5, seed=81)[0]).clamp(0, 1))
        mask = synth.random_mask(shape, 0.15, seed=82) if walls else None
        kw = dict(tau_l=0.8, tau_h=1.1 if contrast else 0.8, sigma=0.01, D=0.1, rho_l=0.6 if contrast else 1.0,
                  rho_h=1.4 if contrast else 1.0)
        two = dict(rho_l=kw["rho_l"], rho_h=kw["rho_h"], tau_l=kw["tau_l"], tau_h=kw["tau_h"], sigma=0.01, width=4.0,
                   diffusivity=0.1, body_accel=(1e-6, 0.0, 2e-6))
        s = _solver(None, shape=shape, lattice=19, storage="f32", two_component=two, mask=mask, force=(1e-6, -1e-6, 0.0))
        s.set_moments(M0.cuda(), phi0.cuda())
        s.step(STEPS)
        want, wphi = oracle.phase.run(oracle.D3Q19, as_f32_exact(M0), phi0, STEPS, kw["tau_l"], kw["tau_h"], 0.01, 4.0, 0.1,
                                      rho_l=kw["rho_l"], rho_h=kw["rho_h"], body=(1e-6, -1e-6, 0.0), solid=mask,
                                      body_accel=(1e-6, 0.0, 2e-6))
        err = _errors(s.moments(), want)
        assert max(err.values()) < TOL["f32"], (shape, err)
        assert (s.phi().cpu() - wphi).abs().max() < TOL["f32"] * wphi.abs().max(), shape
