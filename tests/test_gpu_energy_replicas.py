"""Energies of batches whose replicas are all, some or none of one block of the energy
sums (-m gpu): one pass or two, the same bits as each replica alone."""
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


@pytest.mark.parametrize("mols", [(2,), (204, 2, 2, 204), (205, 2, 410, 204), (205, 410), (2, 2, 205)])
def test_energies_of_a_batch_are_those_of_its_replicas(mols):
    reps = [methane(n, seed=20 + k) for k, n in enumerate(mols)]
    kw = dict(cr_enabled=False, kappa_fixed=1.5, max_steps=3)
    out = []
    for s in [W.concat(reps)] + reps:
        g = M.IonisingMD(s, W.atomic_data(8.0), **kw)
        g.step(2)
        out.append(g.energies())
        ek, ep, _ = g.energies()                       # again: nothing is left over
        assert np.array_equal(ek, out[-1][0]) and np.array_equal(ep, out[-1][1])
        g.close()
    for k in (0, 1):
        assert np.array_equal(out[0][k], np.concatenate([o[k] for o in out[1:]]))
    assert out[0][2] == sum(o[2] for o in out[1:]) and (out[0][0] > 0).all()
