"""Blocks of 12 warps pinned (-m gpu): launched as the blocks that fill an SM beside the
LJ table, 4, 10 or 20 warps by its size, with the forces of every other shape bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import water

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


# 9, 28, 43, 46, 47, 67 and 119 type states; more atoms than the instance for few chunks takes
@pytest.mark.parametrize("z", [(8,), (18, 8), (32, 9), (32, 12), (32, 13), (32, 32), (32, 32, 32, 19)])
def test_pinned_blocks_of_12_warps(z):
    z = np.array(z, np.int32)
    s, rc = water(6_000)
    rng = np.random.default_rng(len(z))
    sp = rng.integers(0, len(z), s.n_atoms).astype(np.uint8)
    s = dataclasses.replace(s, species=sp, q0=rng.integers(0, np.minimum(z[sp], 4) + 1).astype(np.uint8))
    kw = dict(sigma0=np.full(len(z), 0.25), eps0=np.full(len(z), 0.2), mass=z * 2.0, r_cut=rc, cr_enabled=False,
              kappa_fixed=3.0, max_steps=4, list_skin_nm=0.1)
    out = []
    for shape in ({}, dict(pair_warps=12), dict(pair_warps=12, pair_blocks_per_sm=1), dict(pair_warps=8)):
        g = M.IonisingMD(s, W.atomic_data(8.0, z=z), launch_shape=shape, **kw)
        g.step(3)
        e = g.energies()
        out.append([g.get_state(M.MD_FIELD_X | M.MD_FIELD_F), e])
        g.close()
    for o in out[1:]:
        assert all(np.array_equal(out[0][0][k], o[0][k]) for k in ("x", "f"))
        assert np.array_equal(out[0][1][1], o[1][1]) and out[0][1][2] == o[1][2]
