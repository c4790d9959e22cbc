"""The kernels that evaluate every face once (kernels_simt.cu, kernels_vjp.cu, kernels_ns.cu), on meshes
above every size rule of the dispatch: tiles of 6 and of 32 elements with a ragged last one, an odd
number of elements (at P2 in FP32 its tile ends in the middle of a 16-byte access), all orders and
both fluxes.  The smaller meshes of the other files meet the kernels below those rules.

Bars.  FP64: 1e-12 of the term scale for the residual, 1e-11 of the largest entry for the VJP, the bars of
test_gpu_parity and test_gpu_adjoint.  FP32: 1e-4 of the term scale (test_gpu_parity derives it), 1e-4
of the largest entry for the VJP.  A stage adds dt R to the state, so its error is dt times the
residual's plus the rounding of the FP32 state: half an ulp of the stored input and of the result,
2^-23 of the largest value together; a step of three stages, whose weights sum to one, three times both.
"""
import numpy as np
import pytest

from oracle.dg import Problem
from paper_2209_01877_gb300 import dg
from paper_2209_01877_gb300 import inputs as I

from gpu_helpers import FLUX, PREC, max_rel_err, residual_term_scale, torch_cuda

pytestmark = pytest.mark.gpu
MU = 0.05


def _walled(ne):
    """The first ne tetrahedra of a jittered box in lattice order, every exposed face a wall."""
    m = I.make_box_mesh((13, 13, 12), periodic=(False, False, False), jitter=0.1, shuffle_elements=False)
    return m.tet_vid[:ne], m.tet_xyz[:ne], np.ones((ne, 4), dtype=np.int8)


def _periodic(dims):
    m = I.make_box_mesh(dims, jitter=0.1)
    return m.tet_vid, m.tet_xyz, None


def _mesh(arrays, p, flux, precision, order=dg.DG_ORDER_MORTON):
    return dg.Mesh(*arrays, order=p, precision=PREC[precision], flux=FLUX[flux], renumber=order)


def _state(P):
    """A smooth wave (P: an oracle problem or a library mesh, for its projection), every element scaled
    by up to 2%, and its energy by up to 1% more: all faces carry jumps, in the wave speeds too (no tie
    for the derivative of their maximum), and the residual is of the size of its terms."""
    def field(x):
        U = I.entropy_wave(0.5 * x)
        U[..., 3] += 0.1 * np.sin(2 * np.pi * x[..., 0])
        return U
    xi = 2.0 * np.random.default_rng(5).random((2, P.ne, 1)) - 1.0
    U = P.project(field) * (1.0 + 0.02 * xi[0, :, None])
    U[:, 4] *= 1.0 + 0.01 * xi[1]
    return U


# P1 stages take these kernels on larger meshes than P2 and P3 do (capi.cpp)
@pytest.mark.parametrize("p,dims", [(1, (22, 23, 23)), (2, (11, 11, 12)), (2, (13, 13, 12)), (3, (11, 11, 12)),
                                    (3, (13, 13, 12))])
@pytest.mark.parametrize("flux", ["rusanov", "roe"])
def test_fp32_stage(p, dims, flux):
    arrays = _periodic(dims)
    P = Problem(*arrays, p=p, flux=flux)
    U = _state(P)
    R = P.residual(U)
    scale = max(residual_term_scale(P, U))
    dt = P.stable_dt(U, 1.0)
    M = _mesh(arrays, p, flux, "fp32")
    dg.dg_set_state(M.handle, U)
    dg.dg_rk_stage(M.handle, 1, dt)
    # stage 1 leaves U1 = U0 + dt R in a buffer of its own; stages 2 and 3 with dt = 0 bring a sixth of
    # its step to the state: 1/3 U0 + 2/3 (3/4 U0 + 1/4 U1)
    dg.dg_rk_stage(M.handle, 2, 0.0)
    dg.dg_rk_stage(M.handle, 3, 0.0)
    out = np.empty_like(U)
    dg.dg_get_state(M.handle, out)
    dg.dg_sync_status(M.handle)
    bar = dt * 1e-4 * scale / 6.0 + 3 * 2.0 ** -23 * np.abs(U).max()
    assert np.abs(dt * R / 6.0).max() > 100 * bar
    assert np.abs(out - (U + dt * R / 6.0)).max() < bar
    # one step of the fused stages against the same stages as a residual and an update
    dt = P.stable_dt(U, 0.3)
    dg.dg_set_state(M.handle, U)
    dg.dg_rk3_step(M.handle, dt, 1)
    dg.dg_get_state(M.handle, out)
    two = np.empty_like(U)
    dg.dg_set_state(M.handle, U)
    dg.dg_ns_rk3_step(M.handle, dt, 1, 0.0)
    dg.dg_get_state(M.handle, two)
    assert np.abs(out - two).max() <= 4 * 2.0 ** -23 * np.abs(U).max()
    M.close()


@pytest.mark.parametrize("ne", [8193, 9731])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_fp32_ns_step_walled_odd(p, ne):
    arrays = _walled(ne)
    P = Problem(*arrays, p=1, flux="roe")   # for the term scale
    out = {}
    for precision in ("fp64", "fp32"):
        M = _mesh(arrays, p, "roe", precision)
        if precision == "fp64":
            U = _state(M)
            dg.dg_set_state(M.handle, U)
            dt = dg.dg_stable_dt(M.handle, 0.1)
        dg.dg_set_state(M.handle, U)
        dg.dg_ns_rk3_step(M.handle, dt, 1, MU)
        out[precision] = np.empty_like(U)
        dg.dg_get_state(M.handle, out[precision])
        dg.dg_sync_status(M.handle)
        M.close()
    scale = max(residual_term_scale(P, U))
    step = np.abs(out["fp64"] - U).max()
    bar = 3 * (dt * 1e-4 * scale + 2.0 ** -23 * np.abs(U).max())
    assert step > 20 * bar
    assert np.abs(out["fp32"] - out["fp64"]).max() < bar


@pytest.mark.parametrize("p", [1, 2, 3])
def test_fp32_inviscid_ns_step_is_the_euler_step(p):
    """dg_rk3_step and dg_ns_rk3_step with mu = 0 may sum the Euler lines in two orders: each within the FP32
    bar of the residual, so twice that of a step apart."""
    arrays = _walled(9731)
    scale_of = Problem(*arrays, p=1, flux="roe")
    M = _mesh(arrays, p, "roe", "fp32")
    U = _state(M)
    dg.dg_set_state(M.handle, U)
    dt = dg.dg_stable_dt(M.handle, 0.3)
    out = []
    for step in (lambda: dg.dg_rk3_step(M.handle, dt, 1), lambda: dg.dg_ns_rk3_step(M.handle, dt, 1, 0.0)):
        dg.dg_set_state(M.handle, U)
        step()
        out.append(np.empty_like(U))
        dg.dg_get_state(M.handle, out[-1])
    bar = 2 * 3 * (dt * 1e-4 * max(residual_term_scale(scale_of, U)) + 2.0 ** -23 * np.abs(U).max())
    assert np.abs(out[0] - U).max() > 20 * bar
    assert np.abs(out[0] - out[1]).max() < bar
    M.close()


@pytest.mark.parametrize("p", [2, 3])
def test_fp32_adjoint_of_a_walled_step(p):
    """The stages that the adjoint recomputes on a mesh with boundary faces against those of the step it
    differentiates: FP32 rounding of the states (1e-7 of them) through second derivatives of order one,
    within the FP32 bar of the VJP.  Reference: the FP64 mesh, whose stages have one form."""
    torch = torch_cuda()
    arrays = _walled(9731)
    V = {}
    for precision in ("fp64", "fp32"):
        M = _mesh(arrays, p, "roe", precision)
        if precision == "fp64":
            U = _state(M)
            dg.dg_set_state(M.handle, U)
            dt = dg.dg_stable_dt(M.handle, 0.1)
            Ud, lam = torch.from_numpy(U).cuda(), torch.from_numpy(I.random_directions(U.shape, 1)[0]).cuda()
        out = torch.full_like(Ud, float("nan"))
        dg.dg_rk3_step_vjp(M.handle, Ud, dt, lam, out)
        V[precision] = out.cpu().numpy()
        M.close()
    assert max_rel_err(V["fp32"], V["fp64"]) < 1e-4


@pytest.mark.parametrize("p,flux", [(1, "roe"), (2, "rusanov"), (3, "roe")])
def test_residual_and_vjp_ragged(p, flux):
    """FP64 against the oracle, FP32 against FP64, at 9,731 elements with walls."""
    torch = torch_cuda()
    arrays = _walled(9731)
    P = Problem(*arrays, p=p, flux=flux)
    U = _state(P)
    lam = I.random_directions(U.shape, 1)[0]
    Ud, lamd = torch.from_numpy(U).cuda(), torch.from_numpy(lam).cuda()
    R, V = {}, {}
    for precision in ("fp64", "fp32"):
        M = _mesh(arrays, p, flux, precision)
        out = torch.full_like(Ud, float("nan"))
        dg.dg_residual(M.handle, Ud, out)
        dg.dg_sync_status(M.handle)
        R[precision] = out.cpu().numpy()
        out.fill_(float("nan"))
        dg.dg_residual_vjp(M.handle, Ud, lamd, out)
        V[precision] = out.cpu().numpy()
        M.close()
    ref, scale = P.residual(U), residual_term_scale(P, U)
    assert max_rel_err(R["fp64"], ref, term_scale=scale) < 1e-12
    assert max_rel_err(R["fp32"], ref, term_scale=scale) < 1e-4
    assert max_rel_err(V["fp64"], P.vjp(U, lam)) < 1e-11
    assert max_rel_err(V["fp32"], V["fp64"]) < 1e-4


@pytest.mark.parametrize("k", [2, 6])
@pytest.mark.parametrize("p", [1, 2, 3])
def test_partition_of_smaller_tiles_is_bitwise(p, k):
    """FP64: the whole mesh takes tiles of 32 elements, its halves tiles of 6 and its sixths at P3 four
    warps per tile; an element's arithmetic does not depend on any of it."""
    torch = torch_cuda()
    arrays = _periodic((13, 13, 12))
    M = _mesh(arrays, p, "roe", "fp64", order=dg.DG_ORDER_HILBERT)
    U = torch.from_numpy(_state(M)).cuda()
    R, Rp = torch.empty_like(U), torch.full_like(U, float("nan"))
    dg.dg_residual(M.handle, U, R)
    part = dg.dg_partition_create(M.handle, k)
    try:
        dg.dg_partition_residual(part, U, Rp)
        np.testing.assert_array_equal(Rp.cpu().numpy(), R.cpu().numpy())
    finally:
        dg.dg_partition_destroy(part)
        M.close()
