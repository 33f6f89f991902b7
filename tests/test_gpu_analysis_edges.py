"""Edges of the analysis kernels (-m gpu): replicas around the block size of
the energy sums, and fragment radii from far inside the list's radius (where
cluster boxes decide what is looked at) to the cutoff itself."""
import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def test_energy_sums_around_the_block_size():
    """Replicas of 10, 1,020, 1,025, 2,050 and 3,080 atoms (blocks of 1,024):
    kinetic energies against numpy to the rounding of a sum of that many
    terms, and both energies of a replica alone equal to its slot's, bit for bit."""
    reps = [methane(n, seed=60 + k) for k, n in enumerate((2, 204, 205, 410, 616))]
    for k, r in enumerate(reps):
        r.seed[:] = 70 + k
    kw = dict(cr_enabled=False, kappa_fixed=1.5, max_steps=5)
    atom = W.atomic_data(8.0)
    s = W.concat(reps)
    g = M.IonisingMD(s, atom, **kw)
    ek, ep, _ = g.energies()
    g.close()
    for k, r in enumerate(reps):
        terms = 0.5 * W.MASS[r.species] * (r.v ** 2).sum(1)
        assert abs(ek[k] - terms.sum()) <= 4 * np.finfo(float).eps * np.log2(len(terms)) * terms.sum()
        one = M.IonisingMD(r, atom, **kw)
        ek1, ep1, _ = one.energies()
        one.close()
        assert ek1[0] == ek[k] and ep1[0] == ep[k]


@pytest.mark.parametrize("r_frag", [0.05, 0.3, 0.7, 1.05, 1.2])
@pytest.mark.parametrize("skin", [0.0, 0.1])
def test_fragment_radius_range_matches_oracle(oracle_mod, skin, r_frag):
    """A thin gas of atoms (a methane cluster spread out three times) that
    has moved away from the list's build positions."""
    from test_gpu_fragments import _check
    s = methane(240, charge_frac=0.5)
    s.x *= 3.0
    s.v *= 20.0
    g = M.IonisingMD(s, W.atomic_data(8.0), r_cut=1.2, cr_enabled=False, kappa_fixed=1.0, max_steps=20, list_skin_nm=skin)
    g.step(12)
    _check(oracle_mod, g, s, min(r_frag, 1.2 - 2e-3) if r_frag >= 1.2 else r_frag)
    g.close()
