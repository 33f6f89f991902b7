"""State exchange (-m gpu): arrays split, joined and checked on the device, at
sizes around a block of 256 atoms; a refused field is not stored."""
import dataclasses

import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _first(s, n):
    return dataclasses.replace(s, x=s.x[:n], v=s.v[:n], species=s.species[:n], fragment=s.fragment[:n], q0=s.q0[:n],
                               replica_offset=np.array([0, n], np.int32))


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1025])
@pytest.mark.parametrize("skin", [0.0, 0.1])
def test_round_trip_and_refusals(n, skin):
    s = _first(methane(210), n)
    g = M.IonisingMD(s, W.atomic_data(8.0), r_cut=1.2, max_steps=5, list_skin_nm=skin)
    rng = np.random.default_rng(n)
    x = s.x + rng.uniform(-0.01, 0.01, s.x.shape)
    v = rng.normal(size=s.v.shape)
    q = (rng.random(n) < 0.5).astype(np.uint8)
    h = np.zeros(n, np.uint8)
    h[-1] = 1 if W.Z[s.species[-1]] > 2 else 0
    xl = x + 0.01
    fields = M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_Q | M.MD_FIELD_H | M.MD_FIELD_XLIST
    good = dict(x=x, v=v, q=q, h=h, x_list=xl)
    g.set_state(fields, **good)
    st = g.get_state(M.MD_FIELD_ALL)
    for k in ("x", "v", "q", "h"):
        assert np.array_equal(st[k], good[k]), k
    assert np.array_equal(st["x_list"], xl if skin > 0 else x)
    for name, bad in (("x", np.nan), ("x", np.inf), ("v", -np.inf), ("x_list", np.nan)):
        if name == "x_list" and skin == 0:
            continue
        for at in (0, n - 1):
            a = good[name].copy()
            a[at, 2] = bad
            with pytest.raises(M.MDError) as e:
                g.set_state({"x": M.MD_FIELD_X, "v": M.MD_FIELD_V, "x_list": M.MD_FIELD_XLIST}[name], **{name: a})
            assert e.value.status == M.MD_ERR_INVALID_ARG
    for name, bit, val in (("q", M.MD_FIELD_Q, 33), ("h", M.MD_FIELD_H, 2)):
        a = good[name].copy()
        a[n - 1] = val
        with pytest.raises(M.MDError) as e:
            g.set_state(bit, **{name: a})
        assert e.value.status == M.MD_ERR_INVALID_ARG
    after = g.get_state(M.MD_FIELD_X | M.MD_FIELD_V | M.MD_FIELD_Q | M.MD_FIELD_H)
    for k in ("x", "v", "q", "h"):
        assert np.array_equal(after[k], good[k]), k
    g.close()
