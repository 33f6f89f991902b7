"""Pinned launch shapes of the FP64 force kernel, and LJ tables that decide how many
warps its blocks hold (-m gpu): three blocks of 4 warps are accepted up to 30 type
states, 94 states with blocks of 4 warps; the forces are the oracle's, and those of
other shapes bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import force_errors, methane

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _system(z):
    z = np.array(z, np.int32)
    s = methane(120, charge_frac=0.0)
    rng = np.random.default_rng(len(z))
    sp = rng.integers(0, len(z), s.n_atoms).astype(np.uint8)
    q0 = rng.integers(0, np.minimum(z[sp], 6) + 1).astype(np.uint8)
    q0[:len(z)] = z[sp[:len(z)]]                       # the last state of a species too
    s = dataclasses.replace(s, species=sp, q0=q0)
    kw = dict(sigma0=rng.uniform(0.2, 0.3, len(z)), eps0=rng.uniform(0.1, 0.5, len(z)), mass=rng.uniform(1.0, 40.0, len(z)))
    return s, W.atomic_data(8.0, z=z), kw


def _forces(s, atom, kw, **more):
    g = M.IonisingMD(s, atom, r_cut=1.2, cr_enabled=False, kappa_fixed=3.0, max_steps=2, **kw, **more)
    f = g.get_state(M.MD_FIELD_F)["f"]
    g.close()
    return f


# 28, 30, 55, 56, 93, 94 type states
@pytest.mark.parametrize("z", [(18, 8), (18, 10), (32, 21), (32, 22), (32, 32, 26), (32, 32, 27)])
def test_fp64_shapes(oracle_mod, z):
    s, atom, kw = _system(z)
    f = _forces(s, atom, kw, precision="fp64", launch_shape=dict(pair_warps=4))
    ora = oracle_mod.OracleMD(s, atom, r_cut=1.2, cr_enabled=False, kappa_fixed=3.0, **kw)
    rms, mx = force_errors(f, ora.F)
    assert rms <= 1e-9, (rms, mx)                      # the tolerance of the parity tests
    assert np.array_equal(f, _forces(s, atom, kw, precision="fp64"))
    if len(z) == 2 and sum(z) + 2 <= 30:
        assert np.array_equal(f, _forces(s, atom, kw, precision="fp64", launch_shape=dict(pair_warps=4, pair_blocks_per_sm=3)))


# 41, 42 and 90 type states: both sides of the line between blocks of 8 and 4 warps, and the last of 4
@pytest.mark.parametrize("z", [(32, 7), (32, 8), (32, 32, 23)])
def test_fp64_hybrid_shapes(z):
    s, atom, kw = _system(z)
    f = [_forces(s, atom, kw, precision="fp64", screening="hybrid", launch_shape=sh) for sh in ({}, dict(pair_warps=4))]
    assert np.array_equal(f[0], f[1]) and np.abs(f[0]).max() > 0


def test_fp64_pins_beyond_the_limits_are_refused():
    s, atom, kw = _system((18, 8))
    for shape in (dict(pair_warps=4, pair_blocks_per_sm=4), dict(pair_warps=8, pair_blocks_per_sm=2)):
        with pytest.raises(M.MDError) as e:
            _forces(s, atom, kw, precision="fp64", launch_shape=shape)
        assert e.value.status == M.MD_ERR_INVALID_ARG


def test_pinned_blocks_choose_warps_that_fit():
    """128 type states, mixed: blocks of 12 warps and the table do not fit an SM."""
    s, atom, kw = _system((32, 32, 32, 28))
    assert np.array_equal(_forces(s, atom, kw), _forces(s, atom, kw, launch_shape=dict(pair_blocks_per_sm=1)))
