"""What walls add to the workspace: one byte a site for the mask, and the block sums of the rows near them. Only
the masked form of the axis-separated kernel (lattices below 2^20 sites in FP32 and FP64) also holds four bytes of
links a site."""
import ctypes

import pytest

from paper_2609_09160_gb300 import _lbf, build

MIB = 2 ** 20


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()


def _bytes(walls, n, storage, lattice=19, two=False):
    p = _lbf.lbf_params()
    p.lattice, p.nx, p.ny, p.nz, p.storage, p.tau = lattice, n, n, n, storage, 0.8
    if two:
        p.two_component = 1
        p.rho_l = p.rho_h = p.tau_l = p.tau_h = 1.0
        p.width, p.sigma, p.diffusivity = 4.0, 0.03, 0.1
    mask = (ctypes.c_uint8 * 1)()
    if walls:
        p.mask = ctypes.addressof(mask)
    return _lbf.lbf_workspace_bytes(p)


@pytest.mark.parametrize("lattice", [19, 27, 127])
@pytest.mark.parametrize("storage", [_lbf.LBF_F64, _lbf.LBF_F32, _lbf.LBF_F16, _lbf.LBF_BF16])
def test_walls_of_large_lattices_add_a_byte_a_site(storage, lattice):
    for n in (102, 256, 512):
        more = _bytes(True, n, storage, lattice) - _bytes(False, n, storage, lattice)
        assert more < 1.25 * n ** 3 + MIB, (n, more)  # a block sums 64 bytes for at least 480 sites, twice


@pytest.mark.parametrize("storage", [_lbf.LBF_F16, _lbf.LBF_BF16])
def test_walls_of_small_16_bit_lattices_add_a_byte_a_site(storage):
    more = _bytes(True, 96, storage) - _bytes(False, 96, storage)
    assert 96 ** 3 <= more < 96 ** 3 + MIB


def test_two_component_walls_add_a_byte_a_site():
    more = _bytes(True, 160, _lbf.LBF_F32, two=True) - _bytes(False, 160, _lbf.LBF_F32, two=True)
    assert more < 1.25 * 160 ** 3 + MIB


def test_links_where_they_are_used():
    n = 96
    more = _bytes(True, n, _lbf.LBF_F32) - _bytes(False, n, _lbf.LBF_F32)
    assert 5 * n ** 3 <= more < 5.25 * n ** 3 + MIB
