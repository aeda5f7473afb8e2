"""Overlapped launches: on lattices below 2^23 sites a step's kernels may start while the kernel before them in
the stream still runs. Steps issued back to back give, bit for bit, what the same steps give with the stream
synchronised after each one: single-phase (both load paths, walls, force fields, both step kernels), two
components, the adjoint; on two streams at once, with another library's kernel between two steps, and replayed
from a captured graph."""
import os

import pytest
import torch

import synth
from paper_2609_09160_gb300 import Solver

pytestmark = pytest.mark.gpu
STEPS = 40


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


TWO = dict(rho_l=1.0, rho_h=1.0, tau_l=0.8, tau_h=0.8, sigma=0.01, width=4.0, diffusivity=0.1)
CONTRAST = dict(TWO, rho_l=0.6, rho_h=1.4, tau_h=1.1, body_accel=(1e-6, 0.0, 2e-6))
CASES = [
    dict(lattice=19, storage="f32", shape=(40, 48, 64)), dict(lattice=19, storage="f32", shape=(17, 30, 37)),
    dict(lattice=19, storage="f32", shape=(40, 48, 64), kernel="cta"), dict(lattice=27, storage="f64", shape=(20, 18, 32)),
    dict(lattice=127, storage="f32", shape=(20, 34, 68)), dict(lattice=19, storage="f16", shape=(40, 48, 64)),
    dict(lattice=19, storage="f32", shape=(40, 48, 64), walls=0.2), dict(lattice=27, storage="f32", shape=(17, 30, 37), walls=0.2),
    dict(lattice=19, storage="f32", shape=(40, 48, 64), field=True), dict(lattice=19, storage="f32", shape=(96, 128, 128)),
    dict(lattice=19, storage="f32", shape=(34, 130, 260), walls="band"), dict(lattice=19, storage="f32", shape=(24, 48, 64), two=TWO),
    dict(lattice=19, storage="f32", shape=(17, 30, 37), two=CONTRAST, walls=0.15),
    dict(lattice=27, storage="f32", shape=(17, 30, 37), two=TWO), dict(lattice=19, storage="f64", shape=(12, 20, 32), two=CONTRAST),
]


def _make(case, seed=30):
    shape, storage = case["shape"], case["storage"]
    dt = torch.float64 if storage == "f64" else torch.float32
    kw = dict(shape=shape, lattice=case["lattice"], storage=storage, tau=0.8, two_component=case.get("two"))
    if "walls" in case:
        kw["mask"] = synth.channel_walls(shape) if case["walls"] == "band" else synth.random_mask(shape, case["walls"], seed=31)
    if case.get("field"):
        kw["force_field"] = synth.random_field(shape, 1e-5, seed=32).to("cuda", dt)
    M0 = (0.2 * synth.random_moments(shape, seed=seed)).to("cuda", dt)
    phi = None
    if "two" in case and case["two"]:
        phi = (0.5 + 0.4 * synth.random_field(shape, 0.5, seed=33)[0]).clamp(0, 1).to("cuda", dt)
    s = _solver(case.get("kernel"), **kw)
    s.set_moments(M0, phi)
    return s


def _state(s, two):
    x = s.new_state()
    s.copy_state(x)
    return [x] + ([s.phi()] if two else [])


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("case", range(len(CASES)))
def test_steps_back_to_back_equal_synchronised_steps(case):
    c = CASES[case]
    a, b = _make(c), _make(c)
    for _ in range(STEPS):
        b.step(1)
        torch.cuda.synchronize()
    torch.cuda.synchronize()
    a.step(STEPS)
    assert _same(_state(a, c.get("two")), _state(b, c.get("two")))
    assert a.reduce() == b.reduce()


def test_adjoint_steps_back_to_back_equal_synchronised_steps():
    shape, n = (24, 40, 64), 20
    F = synth.random_field(shape, 1e-5, seed=34).to("cuda", torch.float32)
    s = Solver(shape, lattice=19, tau=0.8, storage="f32", force_field=F, mask=synth.channel_walls(shape))
    s.set_moments((0.2 * synth.random_moments(shape, seed=35)).cuda())
    g = torch.Generator(device="cuda").manual_seed(36)
    lam0 = torch.empty((10,) + shape, device="cuda").normal_(generator=g)
    got = []
    for wait in (True, False):
        seg = s.new_state(count=n + 1)
        for k in range(n + 1):
            s.copy_state(seg[k])
        lam, other, gF = lam0.clone(), torch.empty_like(lam0), torch.zeros((3,) + shape, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        for k in range(n):
            s.step_state(seg[k], seg[k + 1])
            if wait:
                torch.cuda.synchronize()
        for k in reversed(range(n)):
            s.adjoint_step(seg[k], seg[k + 1], lam, other, gF)
            lam, other = other, lam
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        got.append((seg, lam, gF))
    assert _same(*got)


def test_two_streams_at_once():
    c = CASES[0]
    alone = []
    for seed in (37, 38):
        s = _make(c, seed)
        s.step(STEPS)
        alone.append(_state(s, False))
    streams = [torch.cuda.Stream() for _ in range(2)]
    both = []
    torch.cuda.synchronize()
    for st, seed in zip(streams, (37, 38)):
        with torch.cuda.stream(st):
            both.append(_make(c, seed))
    torch.cuda.synchronize()
    for _ in range(STEPS):
        for s in both:
            s.step(1)
    torch.cuda.synchronize()
    for s, st, want in zip(both, streams, alone):
        with torch.cuda.stream(st):
            got = _state(s, False)
        st.synchronize()
        assert _same(got, want)


def test_foreign_kernel_between_steps():
    """The force field is the caller's: what it holds when a step is issued, written by another library's
    kernel directly before, is what the step takes, and the next step's successor does not disturb it."""
    shape = (40, 48, 64)
    base = synth.random_field(shape, 1e-5, seed=39).to("cuda", torch.float32)
    M0 = (0.2 * synth.random_moments(shape, seed=40)).to("cuda", torch.float32)
    got = []
    for wait in (True, False):
        F = base.clone()
        s = Solver(shape, lattice=19, tau=0.8, storage="f32", force_field=F)
        s.set_moments(M0)
        torch.cuda.synchronize()
        for k in range(STEPS):
            F.mul_(-1.0 if k % 3 else 0.5)
            if wait:
                torch.cuda.synchronize()
            s.step(2)
            if wait:
                torch.cuda.synchronize()
        got.append(_state(s, False))
    assert _same(*got)


@pytest.mark.parametrize("case", [0, 6, 10, 11])
def test_captured_steps_replay(case):
    c = CASES[case]
    two = c.get("two")
    plain = _make(c)
    plain.step(12)
    want = _state(plain, two)
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        s = _make(c)
        s.step(2)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            s.step(2)  # an even number: a replay goes on where the one before ended
        for _ in range(5):
            graph.replay()
        got = _state(s, two)
    torch.cuda.synchronize()
    assert _same(got, want)
