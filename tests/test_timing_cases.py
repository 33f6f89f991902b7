"""The 64-bit reference of the timing cases: what a replica of a batch is given of
the batch's bonded terms."""
import importlib.util
import os

import numpy as np

from paper_2401_03180_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _cases():
    spec = importlib.util.spec_from_file_location("timing_cases", os.path.join(ROOT, "perf", "cases.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def test_each_replica_gets_its_own_bonded_terms(monkeypatch):
    """Every atom index lies within the replica (an index past it would be read on
    the device), the parameter columns stay, and the replicas' terms are the batch's."""
    cases = _cases()
    s = W.with_topology(W.concat([W.methane_cluster(n, k) for k, n in enumerate((3, 1, 5))]))
    seen = []

    def record(x, q, sp, frag, box, kap, ne, hybrid, topo):
        seen.append((len(q), topo))
        return np.zeros((len(q), 3)), 0.0, 0

    monkeypatch.setattr(cases, "_replica_forces", record)
    st = {"x": s.x, "q": s.q0, "n_e": np.zeros(3, np.int64), "e_gas_mev": np.zeros(3, np.int64)}
    cases._forces({"screening": "debye"}, s, st)
    bonds, angles = [], []
    for (n, t), a in zip(seen, s.replica_offset):
        for rows, atoms in ((t.bonds, t.bonds[:, :2]), (t.angles, t.angles[:, :3])):
            assert len(rows) and atoms.min() >= 0 and atoms.max() < n
        bonds.append(t.bonds + [a, a, 0])
        angles.append(t.angles + [a, a, a, 0])
    assert np.array_equal(np.concatenate(bonds), s.topology.bonds)
    assert np.array_equal(np.concatenate(angles), s.topology.angles)
