"""Slots of many cells (-m gpu): a dilute gas of about one atom per cell, whose seven
padding slots a cell bring the slot numbers beyond 2^24, where the padding records of a
cluster coincide in 32 bits."""
import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import force_errors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def test_forces_of_a_gas_beyond_2_to_the_24_slots(oracle_mod):
    m, a, r_cut = 140, 1.25, 1.0
    rng = np.random.default_rng(12)
    x = (np.indices((m, m, m)).reshape(3, -1).T + 0.5) * a + rng.uniform(-0.3, 0.3, (m ** 3, 3))
    n = len(x)
    # eight slots per occupied cell: the grid has at most 2^22 cells, so its edge is below 1.2 nm
    cells = np.unique(np.floor((x - x.min(0)) / 1.2).astype(np.int64) @ np.array([1 << 40, 1 << 20, 1]))
    assert 8 * len(cells) > 1 << 24
    sp = rng.integers(0, len(W.Z), n).astype(np.uint8)
    s = W.Sample(x=x, v=np.zeros((n, 3)), species=sp, fragment=np.arange(n, dtype=np.int32),
                 q0=(rng.random(n) < 0.5).astype(np.uint8), replica_offset=np.array([0, n], np.int32),
                 seed=np.array([5], np.uint64), box=np.zeros((1, 3)), volume=np.array([(m * a) ** 3]))
    atom = W.atomic_data(8.0)
    g = M.IonisingMD(s, atom, r_cut=r_cut, cr_enabled=False, kappa_fixed=1.0, max_steps=2)
    f = g.get_state(M.MD_FIELD_F)["f"]
    pairs = g.energies()[2]
    g.step(1)
    x1 = g.get_state(M.MD_FIELD_X)["x"]
    g.close()
    idx = rng.choice(n, 400, replace=False)
    idx[:200] = np.argsort(x[:, 2])[-200:]                  # the last slots
    rms, mx = force_errors(f[idx], oracle_mod.forces_of_atoms(s, atom, idx, r_cut=r_cut, kappa=1.0))
    assert rms <= 1e-5, (rms, mx)                           # the tolerance of the parity tests
    from scipy.spatial import cKDTree
    t = cKDTree(x)
    lo, hi = ((t.count_neighbors(t, r_cut + d) - n) // 2 for d in (-1e-6, 1e-6))
    assert lo <= pairs <= hi
    dt = 5e-5
    assert np.abs(x1 - (x + 0.5 * dt * dt * f / W.MASS[sp][:, None])).max() <= 1e-9
