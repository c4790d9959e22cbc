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


def rel(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


def calls(M, Ud, ld, out, dt):
    """Every call of a mesh that may allocate, each with a result to compare (out: device scratch of the caller,
    so that nothing but the mesh allocates)."""
    host = np.empty(tuple(Ud.shape))

    def device(f):
        def run():
            out.fill_(float("nan"))
            f()
            return out.cpu().numpy().copy()
        return run

    def stepped(f):
        def run():
            dg.dg_set_state(M.handle, Uh)      # through the staging buffer of host copies
            f()
            dg.dg_get_state(M.handle, host)
            return host.copy()
        return run
    Uh = Ud.cpu().numpy()
    return {
        "step": stepped(lambda: dg.dg_rk3_step(M.handle, dt, 1)),
        "residual": device(lambda: dg.dg_residual(M.handle, Ud, out)),
        "ns_step": stepped(lambda: dg.dg_ns_rk3_step(M.handle, dt, 1, 0.05)),
        "ns_residual": device(lambda: dg.dg_ns_residual(M.handle, Ud, out, 0.05)),
        "vjp": device(lambda: dg.dg_residual_vjp(M.handle, Ud, ld, out)),
        "step_vjp": device(lambda: dg.dg_rk3_step_vjp(M.handle, Ud, dt, ld, out)),
    }


def room():
    """Memory for exactly the buffers that the calls cannot do without, then for a little more at a time: every
    call runs, in any order, and gives what it gives on a mesh with room."""
    m = I.make_box_mesh((12, 11, 11), jitter=0.1)
    M = mesh(m)
    U = torch.from_numpy(state(M)).cuda()
    lam = torch.from_numpy(I.random_directions(U.shape, 1)[0]).cuda()
    dt = 1e-3
    out = torch.empty_like(U)
    ref = {k: f() for k, f in calls(M, U, lam, out, dt).items()}
    nb, nqf, ne, rs = M.nb, M.nqf, M.ne, 8 if PRECISION == "fp64" else 4
    M.close()
    for k in ref:
        assert np.isfinite(ref[k]).all(), k
    base = shim.fake_in_use()
    face = 20 * nqf * ne * rs
    need = ne * (16 + 4 + 4 + 72) + (1 << 20)                                     # connectivity, geometry; tables
    need += ne * 36 if PRECISION == "fp32" else ne * (12 + 96) + 2 * face         # FP32 geometry; FP64 faces
    need += 11 * (5 * nb * ne * rs + 256) + 5 * nb * ne * 8                       # state, work, adjoint; host copies
    need += 15 * nb * ne * rs + 16 * nqf * ne * rs                                # viscous passes
    # the size of one Euler term, |F| |grad lambda|, and of one viscous term, kappa |U| |grad lambda|^2
    E = np.linalg.inv((m.tet_xyz[:, 1:] - m.tet_xyz[:, :1]).transpose(0, 2, 1))
    inv_h = max(np.linalg.norm(E, axis=2).max(), np.linalg.norm(E.sum(1), axis=1).max())
    mean = np.sqrt(6.0) * np.abs(U.cpu().numpy()[:, :, 0])
    speed = (mean[:, 1:4] / mean[:, :1]).max()
    euler_size = inv_h * (mean[:, 4].max() * 1.4 * speed + 0.4 * mean[:, 4].max())
    viscous_size = 0.05 * 1.4 / (0.4 * 0.72) * mean.max() * inv_h ** 2
    names = list(ref)
    for extra in (0.0, 0.5, 1.0, 1.5, 2.0, 3.0, 4.0, 8.0):
        for order in (names, names[::-1]):
            shim.fake_limit(base + need + int(extra * face))
            M = mesh(m)
            got = calls(M, U, lam, out, dt)
            for k in order + order:
                r = got[k]()
                if PRECISION == "fp64":
                    assert np.array_equal(r, ref[k]), (extra, k)
                elif k in ("step", "ns_step"):
                    # two FP32 evaluations, each within 1e-4 of the size of the residual's terms, over three stages
                    size = euler_size + (viscous_size if k == "ns_step" else 0.0)
                    bar = 2 * 3 * (dt * 1e-4 * size + 2.0 ** -23 * np.abs(ref[k]).max())
                    assert np.abs(r - ref[k]).max() < bar, (extra, k, np.abs(r - ref[k]).max(), bar)
                else:
                    assert rel(r, ref[k]) < 1e-4, (extra, k, rel(r, ref[k]))
            M.close()
            shim.fake_limit(2 ** 64 - 1)
            assert shim.fake_in_use() == base and shim.fake_bad_frees() == 0


def streams():
    """An adjoint call on one stream leaves steps on another alone, with room for buffers of its own and
    without."""
    m = I.make_box_mesh((12, 11, 11), jitter=0.1)
    M = mesh(m)
    U = torch.from_numpy(state(M)).cuda()
    lam = torch.from_numpy(I.random_directions(U.shape, 1)[0]).cuda()
    out, ref, got = torch.empty_like(U), torch.empty_like(U), torch.empty_like(U)
    dt, n = 1e-4, 40
    face = 20 * M.nqf * M.ne * 8
    dg.dg_set_state(M.handle, U)
    dg.dg_rk3_step(M.handle, dt, n)
    dg.dg_get_state(M.handle, ref)
    dg.dg_residual_vjp(M.handle, U, lam, out)
    want = out.clone()
    used = shim.fake_in_use()
    M.close()
    torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    for tight in (False, True):
        # without the adjoint's second face buffer, or any room beyond it
        shim.fake_limit(used - face // 2 if tight else 2 ** 64 - 1)
        M = mesh(m)
        for _ in range(3):
            dg.dg_set_state(M.handle, U)
            torch.cuda.synchronize()
            dg.dg_rk3_step(M.handle, dt, n, stream=a)
            for _ in range(4):
                dg.dg_residual_vjp(M.handle, U, lam, out, stream=b)
            dg.dg_get_state(M.handle, got, stream=a)
            torch.cuda.synchronize()
            assert torch.equal(got, ref) and torch.equal(out, want), tight
        M.close()
        shim.fake_limit(2 ** 64 - 1)


{"creation": creation, "room": room, "streams": streams}[CHECK]()
print("CHILD OK")
