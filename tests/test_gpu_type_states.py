"""Forces with many type states (-m gpu): the LJ table grows with their square
and decides how many warps share a block's copy, up to the 128 the interface
allows (mixed) and to tables the FP64 kernel holds with 4-warp blocks."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import force_errors, methane

pytestmark = pytest.mark.gpu
TOL_F = {"mixed": 1e-5, "fp64": 1e-9}   # the tolerances of the parity tests


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


@pytest.mark.parametrize("prec,z", [("mixed", (1,)), ("mixed", (32, 32, 2)), ("mixed", (32, 32, 32, 28)),
                                    ("fp64", (32, 15)), ("fp64", (32, 20)), ("fp64", (32, 32, 2))])
@pytest.mark.parametrize("warps", [0, 4, 8])
def test_forces_with_many_type_states(oracle_mod, prec, z, warps):
    z = np.array(z, np.int32)
    s = methane(120, charge_frac=0.0)
    rng = np.random.default_rng(len(z))
    sp = rng.integers(0, len(z), s.n_atoms).astype(np.uint8)
    q0 = rng.integers(0, np.minimum(z[sp], 6) + 1).astype(np.uint8)
    q0[:len(z)] = z[sp[:len(z)]]                       # the last state of a species too
    s = dataclasses.replace(s, species=sp, q0=q0)
    kw = dict(sigma0=rng.uniform(0.2, 0.3, len(z)), eps0=rng.uniform(0.1, 0.5, len(z)), mass=rng.uniform(1.0, 40.0, len(z)))
    atom = W.atomic_data(8.0, z=z)
    ora = oracle_mod.OracleMD(s, atom, r_cut=1.2, cr_enabled=False, kappa_fixed=3.0, **kw)
    g = M.IonisingMD(s, atom, precision=prec, r_cut=1.2, cr_enabled=False, kappa_fixed=3.0, max_steps=2,
                     launch_shape=dict(pair_warps=warps), **kw)
    f = g.get_state(M.MD_FIELD_F)["f"]
    g.close()
    rms, mx = force_errors(f, ora.F)
    assert rms <= TOL_F[prec], (rms, mx)
