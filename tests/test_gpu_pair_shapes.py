"""Launch shapes of the force kernel beside LJ tables of many type states (-m gpu).

20 warps per SM run as blocks of 4, 10 or 20 by the size of the table a block
copies; forces and pair counts are those of a pinned shape bit for bit, on both sides
of each line, and pins beyond the interface's limits are still refused."""
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


def _system(z):
    s, rc = water(6_000)          # more atoms than the instance for few chunks takes
    assert s.n_atoms > 16_384
    z = np.array(z, np.int32)
    rng = np.random.default_rng(len(z))
    sp = rng.integers(0, len(z), s.n_atoms).astype(np.uint8)
    q0 = rng.integers(0, np.minimum(z[sp], 4) + 1).astype(np.uint8)
    s = dataclasses.replace(s, species=sp, q0=q0)
    kw = dict(sigma0=np.full(len(z), 0.25), eps0=np.full(len(z), 0.2), mass=z * 2.0, r_cut=rc, cr_enabled=False,
              kappa_fixed=3.0, max_steps=4, list_skin_nm=0.1)
    return s, W.atomic_data(8.0, z=z), kw


# 27, 28, 29 type states; 46, 47; 66, 68; 128
@pytest.mark.parametrize("z", [(17, 8), (18, 8), (19, 8), (32, 12), (30, 15), (32, 32), (32, 32, 1), (32, 32, 32, 28)])
def test_default_shape_equals_a_pinned_one(z):
    s, atom, kw = _system(z)
    out = []
    for shape in ({}, dict(pair_warps=4, pair_blocks_per_sm=1)):
        g = M.IonisingMD(s, atom, launch_shape=shape, **kw)
        g.step(3)
        out.append(g.get_state(M.MD_FIELD_X | M.MD_FIELD_F))
        g.close()
    assert np.array_equal(out[0]["f"], out[1]["f"]) and np.array_equal(out[0]["x"], out[1]["x"])


@pytest.mark.parametrize("shape", [dict(pair_warps=4, pair_blocks_per_sm=5), dict(pair_blocks_per_sm=4)])
def test_pins_beyond_the_limits_are_refused(shape):
    s, atom, kw = _system((32, 12))     # 46 type states: four blocks of 4 warps, two of 8
    with pytest.raises(M.MDError) as e:
        M.IonisingMD(s, atom, launch_shape=shape, **kw)
    assert e.value.status == M.MD_ERR_INVALID_ARG
