"""Runs the axis-separated step kernel on odd lattice shapes through the library named by LBF_LIBRARY (the
index-checked LBF_DEBUG build in tests/test_gpu_sep_index_checks.py) and prints one line per case with the status
of lbf_synchronize; exits non-zero if any case fails."""
import os
import sys

import torch

import synth
from paper_2609_09160_gb300 import LBFError, Solver

# rows shorter than a tile, of exactly one tile (FP64 32 columns, else 64), with a moved last tile, by cp.async;
# partial row groups; one plane and several chunks. 16-bit rows are of even length
SHAPES = [(1, 1, 1), (3, 5, 7), (4, 9, 32), (5, 9, 64), (4, 17, 68), (3, 10, 67), (9, 26, 132), (2, 33, 40)]
EVEN = [(1, 1, 2), (3, 5, 8), (5, 9, 64), (4, 17, 72), (3, 10, 66), (9, 26, 136)]
TWO = dict(rho_l=1.0, rho_h=1.0, tau_l=0.9, tau_h=1.1, sigma=0.01, width=3.0, diffusivity=0.1)


def cases():
    for lattice in (19, 27, 127):
        for storage in ("f64", "f32", "f16", "bf16"):
            for kind in ("periodic", "walls", "field", "walls+field"):
                if lattice == 127 and "walls" in kind:
                    continue  # not built: those lattices take the 30-column kernel
                for kernel in ("sep", "sepsmall"):
                    for shape in (EVEN if storage in ("f16", "bf16") else SHAPES):
                        yield lattice, storage, kind, shape, kernel
    for kind in ("two", "two+walls", "contrast", "contrast+walls"):
        for shape in SHAPES:
            yield 19, "f32", kind, shape, "sep"
    for lattice in (19, 27):  # the split step (its clean rows, by either kernel) where it is the default
        for storage in ("f32", "f64"):
            yield lattice, storage, "band", (34, 130, 260), None
            yield lattice, storage, "band+field", (34, 130, 260), None


def run(lattice, storage, kind, shape, kernel):
    os.environ.pop("LBF_KERNEL", None)
    if kernel:
        os.environ["LBF_KERNEL"] = kernel
    cdt = torch.float64 if storage == "f64" else torch.float32
    kw = dict(force=(1e-5, 0.0, 0.0))
    if "walls" in kind:
        kw["mask"] = synth.random_mask(shape, 0.2, seed=5)
    if "band" in kind:
        kw["mask"] = synth.channel_walls(shape)
    if "field" in kind:
        kw["force_field"] = synth.random_field(shape, 1e-5, seed=6).to("cuda", cdt)
    if "two" in kind or "contrast" in kind:
        kw["two_component"] = dict(TWO, rho_l=0.7, rho_h=1.3) if "contrast" in kind else TWO
    s = Solver(shape, lattice=lattice, tau=0.8, storage=storage, **kw)
    assert s.kernels_per_step == (3 if "two_component" in kw else 1) or "band" in kind
    phi = synth.random_field(shape, 0.5, seed=8)[0].abs().clamp(0, 1).to("cuda", cdt) if "two_component" in kw else None
    s.set_moments(synth.random_moments(shape, seed=7).to("cuda", cdt), phi)
    s.step(3)
    s.synchronize()
    assert torch.isfinite(s.moments()).all()


def main():
    bad = 0
    for case in cases():
        try:
            run(*case)
            status = "ok"
        except (LBFError, AssertionError) as e:
            status = f"FAIL {e}"
            bad += 1
        print(case, status, flush=True)
    return 1 if bad else 0


if __name__ == "__main__":
    sys.exit(main())
