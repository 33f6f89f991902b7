"""md_get_state with a missing buffer (-m gpu): the call is refused before any copy is
enqueued, so that no buffer of the caller's is written once it has returned."""
import numpy as np
import pytest
import torch

from paper_2401_03180_gb300 import md as M
from paper_2401_03180_gb300 import workloads as W

from gpu_common import methane

pytestmark = pytest.mark.gpu
VECTORS = [("x", M.MD_FIELD_X), ("x_list", M.MD_FIELD_XLIST), ("v", M.MD_FIELD_V), ("f", M.MD_FIELD_F)]


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    from paper_2401_03180_gb300 import build
    build.build()
    assert torch.cuda.is_available(), "GPU tests need a GPU"


@pytest.mark.parametrize("pending", [False, True])
@pytest.mark.parametrize("missing,bit", VECTORS + [("q", M.MD_FIELD_Q), ("h", M.MD_FIELD_H)])
def test_no_buffer_is_written_when_another_is_missing(missing, bit, pending):
    s = methane(300)
    g = M.IonisingMD(s, W.atomic_data(8.0), cr_enabled=False, kappa_fixed=1.0, max_steps=4, list_skin_nm=0.1)
    if pending:
        g.step(2, wait=False)
    st, fields, kept = M.MDState(), bit, []
    for name, b in VECTORS:
        if name != missing:
            t = torch.full((s.n_atoms, 3), -7.0, dtype=torch.float64).pin_memory()
            kept.append(t)
            setattr(st, name, t.data_ptr())
            fields |= b
    with pytest.raises(M.MDError) as e:
        M.md_get_state(g.h, st, fields)
    assert e.value.status == M.MD_ERR_INVALID_ARG and f"{missing} buffer missing" in str(e.value)
    torch.cuda.synchronize()
    assert all((t == -7.0).all() for t in kept)
    x = g.get_state(M.MD_FIELD_X)["x"]                 # the handle goes on
    assert np.isfinite(x).all()
    g.close()
