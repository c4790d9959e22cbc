"""Child process of test_gpu_no_room.py: `python no_room_child.py <shim> <check> <precision> <order>`.  The
shim (fake_alloc/limit.c) is loaded first, so that the library's device allocations go through it;
an allocation that it refuses is answered by the host alone."""
import ctypes
import os
import sys

shim = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL)
shim.fake_in_use.restype = ctypes.c_size_t
shim.fake_limit.argtypes = [ctypes.c_size_t]
shim.fake_fail.argtypes = [ctypes.c_long]
shim.fake_calls.restype = shim.fake_bad_frees.restype = ctypes.c_long

import numpy as np   # noqa: E402
import torch         # noqa: E402

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
from paper_2209_01877_gb300 import dg          # noqa: E402
from paper_2209_01877_gb300 import inputs as I   # noqa: E402

CHECK, PRECISION, P = sys.argv[2], sys.argv[3], int(sys.argv[4])
PREC = {"fp64": dg.DG_FP64, "fp32": dg.DG_FP32, "mixed": dg.DG_MIXED_FP16}[PRECISION]
DG_ERR_OOM = 4


def mesh(m):
    return dg.Mesh(m.tet_vid, m.tet_xyz, None, order=P, precision=PREC, flux=dg.DG_ROE, renumber=dg.DG_ORDER_MORTON)


def state(M):
    return M.project(lambda x: I.isentropic_vortex(x, radius=0.2))


def creation():
    """Every device allocation of dg_mesh_create refused in turn: the mesh is made without what it can do
    without or is refused as out of memory; nothing stays allocated and nothing is freed twice."""
    m = I.make_box_mesh((12, 11, 11), jitter=0.1)   # 8,712 elements: FP32 stages at P2 take the face buffer
    torch.zeros(1, device="cuda")
    M = mesh(m)
    U = state(M)
    dt = 1e-3
    out, ref = np.empty_like(U), np.empty_like(U)

    def step(M, to):
        dg.dg_set_state(M.handle, U)
        dg.dg_rk3_step(M.handle, dt, 1)
        dg.dg_get_state(M.handle, to)
    step(M, ref)
    M.close()
    base, calls = shim.fake_in_use(), shim.fake_calls()
    M = mesh(m)
    n = shim.fake_calls() - calls
    M.close()
    assert n > 5 and shim.fake_in_use() == base, (n, shim.fake_in_use() - base)
    made = 0
    for k in range(n):
        shim.fake_fail(k)
        try:
            M = mesh(m)
        except dg.DGError as e:
            assert e.status == DG_ERR_OOM, str(e)
            M = None
        shim.fake_fail(-1)
        if M is not None:
            made += 1
            step(M, out)
            assert np.abs(out - ref).max() <= 4 * 2.0 ** -23 * np.abs(U).max()
            M.close()
        assert shim.fake_in_use() == base, (k, shim.fake_in_use() - base)
        assert shim.fake_bad_frees() == 0, (k, shim.fake_bad_frees())
    print("allocations", n, "made without", made)


{"creation": creation}[CHECK]()
print("CHILD OK")
