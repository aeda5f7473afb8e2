"""FP64 steps of the axis-separated kernel against extended precision (numpy.longdouble): what many steps add up
to is rounding, not a factor. The kernel's sums are in units of the smallest lattice weight, 1/36 or 1/216. Applied
as one rounded FP64 number (relative error 5.6e-17) it would scale p* and u in every step: 2.2e-15 to
2.8e-15 after 50. Without it 50 steps leave their independent roundings: each about 1.6e-16 of a field's norm in
one step, so at most sqrt(50) times that, 1.2e-15, if none were damped."""
import itertools

import numpy as np
import pytest

import synth
from paper_2609_09160_gb300 import Solver

pytestmark = pytest.mark.gpu
L = np.longdouble
SYM = ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))


def _directions(lattice):
    for c in itertools.product((-1, 0, 1), repeat=3):
        n = sum(map(abs, c))
        if lattice == 27 or n < 3:
            yield c, ((L(8) / 27, L(2) / 27, L(1) / 54, L(1) / 216) if lattice == 27 else (L(1) / 3, L(1) / 18, L(1) / 36))[n]


def _step(M, tau, lattice):
    """Collide and stream the moments M (no force, periodic), one direction at a time."""
    p, u, keep = M[0], M[1:4], 1 - 1 / L(tau)
    P = [u[a] * u[b] + keep * (M[4 + i] - u[a] * u[b]) for i, (a, b) in enumerate(SYM)]
    out = np.zeros_like(M)
    for c, w in _directions(lattice):
        f = p - L(1.5) * (P[0] + P[1] + P[2]) + 3 * (c[0] * u[0] + c[1] * u[1] + c[2] * u[2])
        for i, (a, b) in enumerate(SYM):
            f = f + (L(4.5) if a == b else L(9)) * c[a] * c[b] * P[i]
        f = np.roll(w * f, (c[2], c[1], c[0]), (0, 1, 2))
        out[0] += f
        for a in range(3):
            out[1 + a] += c[a] * f
        for i, (a, b) in enumerate(SYM):
            out[4 + i] += c[a] * c[b] * f
    out[4:7] -= out[0] / 3
    return out


@pytest.mark.parametrize("lattice", [19, 27])
@pytest.mark.parametrize("shape", [(6, 8, 32), (5, 7, 12)])
def test_many_fp64_steps_against_extended_precision(lattice, shape):
    if np.finfo(L).eps > 1e-18:
        pytest.skip("longdouble is no wider than double here")
    M0 = synth.random_moments(shape, seed=101)
    s = Solver(shape, lattice=lattice, tau=0.8, storage="f64")
    s.set_moments(M0.cuda())
    s.step(50)
    got = s.moments().cpu().numpy()
    want = M0.numpy().astype(L)
    for _ in range(50):
        want = _step(want, 0.8, lattice)
    for name, sl in (("p", slice(0, 1)), ("u", slice(1, 4))):
        err = float(np.linalg.norm((got[sl] - want[sl]).astype(float)) / np.linalg.norm(want[sl].astype(float)))
        assert err < 1.2e-15, (name, err)
