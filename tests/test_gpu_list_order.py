"""Light chunks apart (-m gpu): buffered lists of up to 8,192 super-clusters keep the
chunks of few tiles at the end of the chunk table.  Forces, trajectories and pair
counts of a replica alone (ordered list) and among thousands of others (plain list) are
the same bits, also where the list starts too small and grows, and with another launch
shape; the analyses read the ordered list too."""
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


def _molecule(seed):
    s = methane(2, seed=seed % 8)
    return dataclasses.replace(s, x=s.x[:5], v=s.v[:5], species=s.species[:5], fragment=s.fragment[:5], q0=s.q0[:5],
                               replica_offset=np.array([0, 5], np.int32), seed=np.array([100 + seed], np.uint64))


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("kind", ["cluster", "box"])
def test_replica_alone_and_among_thousands(prec, kind):
    one, rc = (methane(1_200, seed=5), 1.2) if kind == "cluster" else water(2_000)
    kw = dict(precision=prec, r_cut=rc, cr_enabled=False, kappa_fixed=2.0, max_steps=8, list_skin_nm=0.1)
    atom = W.atomic_data(8.0)
    out = []
    for s, extra in ((one, {}), (one, dict(list_reserve=1)), (one, dict(launch_shape=dict(pair_warps=4, pair_blocks_per_sm=1))),
                     (W.concat([one] + [_molecule(k) for k in range(8_200)]), {})):
        g = M.IonisingMD(s, atom, **{**kw, **extra})
        g.step(6)
        out.append(g.get_state(M.MD_FIELD_X | M.MD_FIELD_F))
        g.close()
    n = one.n_atoms
    for o in out[1:]:
        assert np.array_equal(out[0]["x"], o["x"][:n]) and np.array_equal(out[0]["f"], o["f"][:n])


def test_analyses_of_an_ordered_list():
    """Pair histograms, pair counts and energies of a box alone (ordered list) and of
    8,200 molecules (plain list) add up to those of both together, whole numbers and bits."""
    box, rc = water(4_000)
    mols = [_molecule(k) for k in range(8_200)]
    res = []
    for s in (box, W.concat(mols), W.concat([box] + mols)):
        g = M.IonisingMD(s, W.atomic_data(6.0), r_cut=rc, cr_enabled=False, kappa_fixed=2.0, max_steps=4, list_skin_nm=0.1)
        res.append((g.rdf(0.9, 60), g.energies()))
        g.close()
    alone, rest, both = res
    assert np.array_equal(alone[0] + rest[0], both[0]) and alone[0].sum() > 0
    assert alone[1][2] + rest[1][2] == both[1][2]
    for k in (0, 1):
        assert np.array_equal(np.concatenate([alone[1][k], rest[1][k]]), both[1][k])
