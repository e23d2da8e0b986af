"""The fixed-point solve and the integer sums at the edges of their ranges, against the oracle:
densities far from 1 (the sums scale with the cell's largest population), gamma near 1 (g far above
f: the sums go back to FP64), a stopping tolerance below the fixed-point resolution (the whole
solve goes back to FP64), block remainders, and lattices one cell thick in both constraint systems
with equal bits.  Tolerance: the parity suite's (1e-11 relative)."""
import numpy as np
import pytest
import torch

from gpu_helpers import TOL, rel_diffs, run_oracle
from oracle import oracle39 as o
from paper_1910_13515_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Lat():
    from paper_1910_13515_gb300 import build
    build.build()
    from paper_1910_13515_gb300.lattice import Lattice
    return Lattice


def check(Lat, s, steps, oracle_kw=None, **over):
    L = Lat.from_setup(s, **over)
    L.step(steps)
    assert L.sync() == 0
    st, fo = run_oracle(s, steps, **(oracle_kw or {}))
    assert fo == 0
    d = rel_diffs(L.read_numpy(), o.macros(st), s.mask, s.gamma)
    assert max(d) <= TOL, d
    return L


@pytest.mark.parametrize("scale", [1e-8, 0.03, 40.0, 1e6])
@pytest.mark.parametrize("thin", [True, False])
def test_density_scales(Lat, scale, thin):
    s = inputs.shear_layer(23, 1.0) if thin else inputs.box(seed=3, shape=(5, 7, 9), mach_rms=0.4)
    s.rho = s.rho * scale
    check(Lat, s, 11)


@pytest.mark.parametrize("gamma", [1.02, 1.3, 1.66])
def test_gamma_moves_the_second_distribution(Lat, gamma):
    s = inputs.shear_layer(19, 0.8)
    s.gamma = gamma
    check(Lat, s, 9)


@pytest.mark.parametrize("tol", [1e-13, 3e-13, 1e-9])
def test_tolerances_on_both_sides_of_the_resolution(Lat, tol):
    s = inputs.box(seed=5, shape=(6, 5, 7), mach_rms=0.5)
    check(Lat, s, 8, {"newton_tol": min(tol, 1e-12)}, newton_tol=min(tol, 1e-12))
    L = Lat.from_setup(s, newton_tol=tol)
    L.step(8)
    assert L.sync() == 0


@pytest.mark.parametrize("cells", [1, 127, 128, 129])
def test_block_remainders(Lat, cells):
    s = inputs.uniform(cells, 1, 1, u=(0.3, -0.2, 0.1))
    s.rho = 1.0 + 0.05 * np.cos(np.arange(cells) * 0.7)
    check(Lat, s, 7)


@pytest.mark.parametrize("scale,gamma", [(1.0, 1.4), (1e-4, 1.4), (1.0, 1.02)])
def test_thin_lattice_has_the_same_bits_in_both_systems(Lat, scale, gamma):
    s = inputs.shear_layer(21, 1.2)
    s.rho, s.gamma = s.rho * scale, gamma
    bufs = []
    for reduce in (1, 0):
        L = Lat.from_setup(s, reduce_2d=reduce)
        L.step(13)
        assert L.sync() == 0
        planes = L.checkpoint()[256:].view(torch.int64).view(130, -1)
        bufs.append(planes[:, :s.ncells])          # without the planes' padding
    assert torch.equal(*bufs)
