"""The step of large systems (-m gpu): from 16 blocks of 32 atoms per SM on, a
thread does an atom's whole step against a table of total rates.  On both sides
of that line, with blocks that span more replicas than a block keeps sums for,
periodic boxes and a ragged last block, every replica has the same state."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane, water

pytestmark = pytest.mark.gpu
FIELDS = (M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_F | M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_PLASMA)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _first5(s):
    return dataclasses.replace(s, x=s.x[:5], v=s.v[:5], species=s.species[:5], fragment=s.fragment[:5], q0=s.q0[:5],
                               replica_offset=np.array([0, 5], np.int32))


@pytest.mark.parametrize("skin,langevin", [(0.0, None), (0.1, None), (0.1, 0.5)])
def test_replicas_step_alike_on_both_sides_of_the_line(skin, langevin):
    import torch
    line = (16 * torch.cuda.get_device_properties(0).multi_processor_count - 1) * 32 + 1   # atoms from which it is taken
    box, rc = water(8_000)
    cluster = methane(300, seed=3)
    rest = (line - 1 - 2 * box.n_atoms - cluster.n_atoms) // 5
    assert rest > 500
    mols = [_first5(methane(2, seed=k)) for k in range(16)]
    reps = [dataclasses.replace(mols[k % 16], seed=np.array([100 + k], np.uint64)) for k in range(rest)]
    reps += [cluster, box, dataclasses.replace(box, seed=np.array([9], np.uint64))]
    more = reps + [dataclasses.replace(mols[5], seed=np.array([7 + k], np.uint64)) for k in range(9)]
    atom = W.atomic_data(8.0, pi_scale=3000.0, ci_scale=10.0)
    kw = dict(r_cut=rc, max_steps=14, t_start_fs=-0.3, list_skin_nm=skin)
    if langevin is not None:
        kw["langevin_g"] = np.full(len(atom.z), langevin)
    out = []
    for part in (reps, more):
        s = W.concat(part)
        assert (s.n_atoms >= line) == (part is more)
        g = M.IonisingMD(s, atom, **kw)
        for k in range(s.n_replicas):
            g.set_pulse([W.Pulse(8.0, 1.0, 4e11 * (1 + k % 7), 0.0)], replica=k)
        g.step(12)
        out.append(g.get_state(FIELDS))
        g.close()
    a, b = out
    n, r = W.concat(reps).n_atoms, len(reps)
    q0 = np.concatenate([x.q0 for x in reps])
    assert (a["q"] != q0).sum() > 200 and (a["q"][:5 * rest] != q0[:5 * rest]).sum() > 20
    for key in ("x", "v", "f", "q", "h"):
        assert np.array_equal(a[key], b[key][:n]), key
    for key in ("n_e", "e_gas_mev", "te_ev", "kappa"):
        assert np.array_equal(a[key], b[key][:r]), key
