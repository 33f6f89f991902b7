"""Refused md_set_state calls in the middle of a run (-m gpu): the run goes on as if the
call had not been made, or, where a field before the refused one has been stored, from
that field with the forces and lists that belong to it."""
import numpy as np
import pytest

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane

pytestmark = pytest.mark.gpu
ALL = M.MD_FIELD_ALL
X, V, Q, H, XL = M.MD_FIELD_X, M.MD_FIELD_V, M.MD_FIELD_Q, M.MD_FIELD_H, M.MD_FIELD_XLIST


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


def _handle(s, prec, skin):
    g = M.IonisingMD(s, W.atomic_data(8.0), precision=prec, cr_enabled=False, kappa_fixed=1.0, max_steps=20, list_skin_nm=skin)
    g.step(6)
    return g


def _refused(g, fields, **arrays):
    with pytest.raises(M.MDError) as e:
        g.set_state(fields, **arrays)
    assert e.value.status == M.MD_ERR_INVALID_ARG


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("skin", [0.0, 0.1])
def test_a_run_goes_on_after_a_refused_call(prec, skin):
    s = methane(150)
    s.v *= 10.0
    n = s.n_atoms
    nan, q_bad = s.x.copy(), s.q0.copy()
    nan[n - 1, 1] = np.nan
    q_bad[n - 1] = 33
    a, b = _handle(s, prec, skin), _handle(s, prec, skin)
    v0 = a.get_state(V)["v"]
    _refused(a, X, x=nan)
    assert np.array_equal(a.get_state(V)["v"], v0)
    _refused(a, V, v=nan)
    _refused(a, Q, q=q_bad)
    _refused(a, H, h=np.full(n, 2, np.uint8))
    one = np.ones(1, np.int64)
    _refused(a, X | M.MD_FIELD_PLASMA, x=s.x, n_e=-one, e_gas_mev=one)
    _refused(a, X | M.MD_FIELD_PLASMA, x=s.x)
    _refused(a, X | M.MD_FIELD_STEP, x=s.x, step=21)
    _refused(a, X | XL, x=s.x)
    a.step(5)
    b.step(5)
    sa, sb = a.get_state(ALL), b.get_state(ALL)
    for k in ("x", "v", "f", "q"):
        assert np.array_equal(sa[k], sb[k]), k
    a.close()
    b.close()


@pytest.mark.parametrize("bad", ["q", "h", "x_list"])
def test_fields_before_the_refused_one_are_stored_with_their_forces(bad):
    s = methane(150)
    n = s.n_atoms
    rng = np.random.default_rng(4)
    x = s.x + rng.uniform(-0.005, 0.005, s.x.shape)
    a, b = _handle(s, "mixed", 0.1), _handle(s, "mixed", 0.1)
    wrong = {"q": np.full(n, 33, np.uint8), "h": np.full(n, 2, np.uint8), "x_list": np.full((n, 3), np.nan)}[bad]
    _refused(a, X | {"q": Q, "h": H, "x_list": XL}[bad], x=x, **{bad: wrong})
    b.set_state(X, x=x)
    for _ in range(2):
        sa, sb = a.get_state(ALL), b.get_state(ALL)
        for k in ("x", "v", "f", "q", "h"):
            assert np.array_equal(sa[k], sb[k]), k
        a.step(4)
        b.step(4)
    a.close()
    b.close()
