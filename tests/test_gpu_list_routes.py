"""Both list builds (-m gpu): the one-kernel build, a block per super-cluster, and the
kernels that give a warp a part of one, taken by samples of many super-clusters and from
32,768 of capacity on.  A vacuum replica reserves about 56 of them, so a batch of some hundred small replicas
takes the second route with few real super-clusters, split into 1, 2, 7 or 14 parts by
the warps of its grid.  Trajectories are those of the replicas alone, bit for bit."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import force_errors, methane, water

pytestmark = pytest.mark.gpu
FIELDS = M.MD_FIELD_X | M.MD_FIELD_F | M.MD_FIELD_Q


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _molecule(k):
    s = methane(2, seed=k % 8)
    return dataclasses.replace(s, x=s.x[:5], v=s.v[:5], species=s.species[:5], fragment=s.fragment[:5], q0=s.q0[:5],
                               replica_offset=np.array([0, 5], np.int32), seed=np.array([100 + k], np.uint64))


def _run(s, steps=4, **kw):
    g = M.IonisingMD(s, W.atomic_data(8.0, pi_scale=1500.0, ci_scale=10.0), max_steps=16, t_start_fs=-0.2, **kw)
    g.set_pulse([W.Pulse(8.0, 10.0, 1e12, 0.0)])
    g.step(steps)
    st = g.get_state(FIELDS)
    g.close()
    return st


def _parts(n_sc, blocks):
    return next(p for p in (1, 2, 7, 14) if p == 14 or p * n_sc >= 8 * blocks)


@pytest.mark.parametrize("skin", [0.0, 0.05])
@pytest.mark.parametrize("n_rep,per_sm,parts", [(1300, 1, 1), (700, 1, 2), (600, 2, 7), (600, 16, 14)])
def test_parts_of_a_super_cluster(n_rep, per_sm, parts, skin):
    import torch
    first = [methane(40, seed=3)] + [_molecule(k) for k in range(8)]
    s = W.concat(first + [_molecule(k) for k in range(8, n_rep)])
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    if n_sm == 152:
        assert _parts(n_rep, per_sm * n_sm) == parts
    b = _run(s, list_skin_nm=skin, launch_shape=dict(list_blocks_per_sm=per_sm))
    for r, one in enumerate(first):
        a = _run(one, list_skin_nm=skin)
        sl = slice(s.replica_offset[r], s.replica_offset[r + 1])
        for k in ("x", "f", "q"):
            assert np.array_equal(a[k], b[k][sl]), (r, k)


@pytest.mark.parametrize("skin", [0.0, 0.05])
def test_more_super_clusters_than_blocks(skin):
    """One and two blocks per SM in the one-kernel build: a block takes several super-clusters."""
    s, rc = water(6_000)
    kw = dict(r_cut=rc - 0.1, list_skin_nm=skin)
    ref = _run(s, **kw)
    for per_sm in (1, 2, 16):
        b = _run(s, launch_shape=dict(list_blocks_per_sm=per_sm), **kw)
        assert all(np.array_equal(ref[k], b[k]) for k in ("x", "f", "q")), per_sm


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_a_cell_of_many_clusters(prec):
    """A droplet of 12,000 atoms in one cell: a warp of the one-kernel build finds more
    j-clusters of a super-cluster than it keeps, and repeats the box tests."""
    one = W.water_droplet(4000, seed=31)
    kw = dict(r_cut=3.1, list_skin_nm=0.04, precision=prec, steps=2)
    assert (one.x.max(0) - one.x.min(0)).max() < 2 * 3.1
    a = _run(one, **kw)
    b = _run(W.concat([one] + [_molecule(k) for k in range(600)]), **kw)
    assert all(np.array_equal(a[k], b[k][:one.n_atoms]) for k in ("x", "f", "q"))


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-5), ("fp64", 1e-9)])      # the tolerances of the parity tests
@pytest.mark.parametrize("m", [15, 16])
def test_a_gas_on_both_sides_of_the_line(oracle_mod, prec, tol, m):
    """One atom a cell, 3,375 and 4,096 super-clusters: one kernel and five."""
    rng = np.random.default_rng(m)
    n, a = m ** 3, 1.26
    x = (np.indices((m, m, m)).reshape(3, -1).T + 0.5) * a + rng.uniform(-0.3, 0.3, (n, 3))
    s = W.Sample(x=x, v=np.zeros((n, 3)), species=rng.integers(0, len(W.Z), n).astype(np.uint8), fragment=np.arange(n, dtype=np.int32),
                 q0=(rng.random(n) < 0.5).astype(np.uint8), replica_offset=np.array([0, n], np.int32), seed=np.array([5], np.uint64),
                 box=np.full((1, 3), m * a), volume=np.array([(m * a) ** 3]))
    atom = W.atomic_data(8.0)
    ora = oracle_mod.OracleMD(s, atom, r_cut=1.2, cr_enabled=False, kappa_fixed=1.0)
    out = []
    for per_sm in (0, 1, 16):
        g = M.IonisingMD(s, atom, r_cut=1.2, precision=prec, cr_enabled=False, kappa_fixed=1.0, max_steps=4,
                         launch_shape=dict(list_blocks_per_sm=per_sm))
        out.append(g.get_state(M.MD_FIELD_F)["f"])
        g.step(3)
        out.append(g.get_state(M.MD_FIELD_X)["x"])
        assert g.timing().build_kernels in ((5, 6, 7, 8) if m == 15 else (9, 10, 11, 12))
        g.close()
    rms, mx = force_errors(out[0], ora.F)
    assert rms <= tol, (rms, mx)
    for k in (2, 4):
        assert np.array_equal(out[0], out[k]) and np.array_equal(out[1], out[k + 1])
