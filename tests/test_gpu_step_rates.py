"""The step against a table of the total rates (-m gpu), taken by large samples whose
table (two entries per replica and type state) is no larger than they are: small replicas
that share a block, more of them than a block keeps sums for, among boxes that make the
sample large enough, each with the state it has alone; and a batch of small replicas
only, which steps without the table."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane, water

pytestmark = pytest.mark.gpu
FIELDS = (M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_F | M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_PLASMA | M.MD_FIELD_COUNTS)


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _first5(s):
    return dataclasses.replace(s, x=s.x[:5], v=s.v[:5], species=s.species[:5], fragment=s.fragment[:5], q0=s.q0[:5],
                               replica_offset=np.array([0, 5], np.int32))


def _reps(n_mol, boxes):
    box, rc = water(8_000)
    mols = [_first5(methane(2, seed=k)) for k in range(16)]
    reps = [dataclasses.replace(mols[k % 16], seed=np.array([100 + k], np.uint64)) for k in range(n_mol)]
    return reps + [methane(40, seed=3)] + [dataclasses.replace(box, seed=np.array([9 + k], np.uint64)) for k in range(boxes)], rc


def _run(sample, atom, rc, skin, langevin):
    kw = dict(r_cut=rc, max_steps=14, t_start_fs=-0.3, list_skin_nm=skin)
    if langevin is not None:
        kw["langevin_g"] = np.full(len(atom.z), langevin)
    g = M.IonisingMD(sample, atom, **kw)
    g.set_pulse([W.Pulse(8.0, 1.0, 1.6e12, 0.0)])
    g.step(12)
    st = g.get_state(FIELDS)
    g.close()
    return st


def _line():
    import torch
    return (16 * torch.cuda.get_device_properties(0).multi_processor_count - 1) * 32 + 1   # atoms of a large sample


def _by_table(s, atom):
    return s.n_atoms >= _line() and 2 * int((atom.z + 1).sum()) * s.n_replicas <= s.n_atoms


@pytest.mark.parametrize("boxes", [4, 0])
@pytest.mark.parametrize("langevin", [None, 0.5])
def test_replicas_of_a_large_sample_step_as_alone(boxes, langevin):
    reps, rc = _reps(900 if boxes else _line() // 5 + 1, boxes)
    atom = W.atomic_data(8.0, pi_scale=3000.0, ci_scale=10.0)
    s = W.concat(reps)
    assert s.n_atoms >= _line() and _by_table(s, atom) == (boxes > 0)
    a = _run(s, atom, rc, 0.0, langevin)
    assert (a["q"] != s.q0).sum() > 100
    for r in [0, 1, 7, 8, 12, 500, 899] + list(range(len(reps) - boxes - 1, len(reps)))[:2]:
        b = _run(reps[r], atom, rc, 0.0, langevin)
        sl = slice(s.replica_offset[r], s.replica_offset[r + 1])
        for key in ("x", "v", "f", "q", "h"):
            assert np.array_equal(a[key][sl], b[key]), (r, key)
        for key in ("n_e", "e_gas_mev", "te_ev", "kappa", "event_counts"):
            assert np.array_equal(a[key][r], b[key][0]), (r, key)


@pytest.mark.parametrize("skin,langevin", [(0.0, None), (0.1, None), (0.1, 0.5)])
def test_with_and_without_the_table(skin, langevin):
    """The same replicas, and with copies of the first ones added (which move alike, so
    that buffered lists are rebuilt at the same steps) until the table would be larger."""
    reps, rc = _reps(900, 4)
    atom = W.atomic_data(8.0, pi_scale=3000.0, ci_scale=10.0)
    s, more = W.concat(reps), W.concat(reps + reps[:500])
    assert _by_table(s, atom) and not _by_table(more, atom) and more.n_atoms >= _line()
    a, b = (_run(x, atom, rc, skin, langevin) for x in (s, more))
    for key in ("x", "v", "f", "q", "h"):
        assert np.array_equal(a[key], b[key][:s.n_atoms]), key
    for key in ("n_e", "e_gas_mev", "te_ev", "kappa", "event_counts"):
        assert np.array_equal(a[key], b[key][:s.n_replicas]), key
