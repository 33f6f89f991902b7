"""The charge update's shortcuts and the last block's reduction (-m gpu).

Events are ruled in or out by FP32 bounds of lam and 1 - e^{-lam} before the FP64
test: charges, K holes, plasma and event counts must stay the oracle's bit for bit
from rates far below one draw's resolution to rates far above one.  Langevin widths
of up to eight species are formed on the lanes beside the plasma scalars: the order
of the species must not matter."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane, water

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


# photo-absorption per step of a carbon atom about 1e-9, 1e-4, 0.05, 0.7 and 50
@pytest.mark.parametrize("scale", [1e-6, 0.1, 50.0, 700.0, 5e4])
@pytest.mark.parametrize("replicas", [1, 3, 60])   # one thread pair per atom; several replicas; one thread per atom
def test_charges_from_tiny_to_huge_rates(oracle_mod, replicas, scale):
    steps = 6
    reps = []
    for k in range(replicas):
        r = methane(300, seed=k)
        r.seed[:] = 40 + k
        reps.append(r)
    s = W.concat(reps)
    atom = W.atomic_data(8.0, pi_scale=scale, ci_scale=10.0 if scale > 1 else 1e-3)
    pulses = [[W.Pulse(8.0, 10.0, 1e12 * (1 + k % 3), 0.0)] for k in range(replicas)]
    g = M.IonisingMD(s, atom, r_cut=1.2, max_steps=steps, t_start_fs=-0.2, list_skin_nm=0.1)
    for k in range(replicas):
        g.set_pulse(pulses[k], replica=k)
    ora = oracle_mod.OracleMD(s, atom, r_cut=1.2, t_start_fs=-0.2, pulses=pulses, n_steps_max=steps, with_forces=False)
    for n in range(steps):
        g.step(1)
        ora.step()
        st = g.get_state(M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_PLASMA | M.MD_FIELD_COUNTS)
        assert np.array_equal(st["q"], ora.q) and np.array_equal(st["h"], ora.h), n
        assert np.array_equal(st["n_e"], ora.n_e) and np.array_equal(st["e_gas_mev"], ora.e_gas), n
        assert np.array_equal(st["event_counts"], ora.counts), n
    g.close()


@pytest.mark.parametrize("replicas", [1, 4, 5])   # reduced by the step kernel, or by the kernel after it
def test_langevin_of_eight_species_in_either_order(replicas):
    z = np.array([1, 6, 7, 8, 11, 15, 16, 20], np.int32)
    mass, g_e = z * 2.0 + 0.5, 0.2 + 0.1 * np.arange(8)
    rng = np.random.default_rng(3)
    reps = []
    for k in range(replicas):
        r = methane(40 + 7 * k, seed=k) if k % 2 else water(300, r_cut=0.6, seed=k)[0]
        sp = rng.integers(0, 8, r.n_atoms).astype(np.uint8)
        r = dataclasses.replace(r, species=sp, q0=np.minimum(r.q0, z[sp]).astype(np.uint8))
        r.seed[:] = 60 + k
        reps.append(r)
    s = W.concat(reps)
    out = []
    for order in (np.arange(8), np.arange(8)[::-1]):
        g = M.IonisingMD(dataclasses.replace(s, species=np.argsort(order)[s.species].astype(np.uint8)),
                         W.atomic_data(8.0, pi_scale=3000.0, z=z[order]), mass=mass[order], langevin_g=g_e[order],
                         sigma0=np.full(8, 0.25), eps0=np.full(8, 0.3), r_cut=0.6, max_steps=12, t_start_fs=-0.3)
        for k in range(replicas):
            g.set_pulse([W.Pulse(8.0, 1.0, 5e11, 0.0)], replica=k)
        g.step(10)
        out.append(g.get_state(M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_Q | M.MD_FIELD_PLASMA))
        g.close()
    assert (out[0]["te_ev"] > 0).all()
    for key in ("x", "v", "q", "n_e", "te_ev", "kappa"):
        assert np.array_equal(out[0][key], out[1][key]), key
