"""The mixed stage kernel starts while the previous stage still runs (launch.cuh), so the state it reads is
written during its own lifetime: no state plane may be read through the read-only path, and a chain
of overlapped stages gives bitwise what the same stages give when each is waited for."""
import os
import re

import numpy as np
import pytest

from paper_2209_01877_gb300 import dg
from paper_2209_01877_gb300 import inputs as I

CSRC = os.path.join(os.path.dirname(os.path.abspath(dg.__file__)), "csrc")


@pytest.mark.parametrize("name", ["kernels_mixed.cu", "mixed_common.cuh"])
def test_state_planes_are_not_read_through_the_read_only_path(name):
    with open(os.path.join(CSRC, name)) as f:
        text = f.read()
    for call in re.findall(r"__ldg\((?:[^()]|\([^()]*\))*\)", text):
        # the operand builders take a state row c; pls holds the state planes
        assert not re.search(r"\bU0?_(hi|lo)\b|\bpls\b|\(?\bc \+ j", call), call


@pytest.mark.gpu
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("conservative", [False, True])
def test_overlapped_stages_are_bitwise_the_waited_ones(p, conservative):
    import torch
    m = I.make_periodic_cube(7, jitter=0.1)   # 2,058 elements: more tiles than SMs, a ragged last one
    M = dg.Mesh(m.tet_vid, m.tet_xyz, None, order=p, precision=dg.DG_MIXED_FP16, flux=dg.DG_ROE,
                renumber=dg.DG_ORDER_HILBERT)
    if conservative:
        dg.dg_set_conservative(M.handle, True)
    U = torch.from_numpy(M.project(lambda x: I.isentropic_vortex(x, radius=0.2))).cuda()
    dg.dg_set_state(M.handle, U)
    dt = dg.dg_stable_dt(M.handle, 0.1)
    chained, waited = torch.empty_like(U), torch.empty_like(U)
    dg.dg_rk3_step(M.handle, dt, 9)           # 8 steps of a graph and one launched stage by stage
    dg.dg_get_state(M.handle, chained)
    dg.dg_set_state(M.handle, U)
    for _ in range(9):
        for stage in (1, 2, 3):
            torch.cuda.synchronize()
            dg.dg_rk_stage(M.handle, stage, dt)
    dg.dg_get_state(M.handle, waited)
    dg.dg_sync_status(M.handle)
    assert not torch.equal(waited, U)
    np.testing.assert_array_equal(chained.cpu().numpy(), waited.cpu().numpy())
    M.close()
