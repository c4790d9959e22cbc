"""The CUDA-core kernels that own (element, variable) rows in tiles of 32 elements: residual, one RK
step and VJP against the oracle at the edges of a tile (1, 31, 32, 33 and 65 elements; an odd number
leaves a part of a 16-byte access at P2 in FP32), with every exposed face a wall, so that boundary and
interior faces meet in one tile.  Tolerances: the parity bars of the residual (FP64 1e-12 and FP32 1e-4
of the term scale) and of the VJP (1e-11, 1e-4 of each quantity's largest entry).
"""
import numpy as np
import pytest

from oracle.dg import Problem
from paper_2209_01877_gb300 import dg
from paper_2209_01877_gb300 import inputs as I

from gpu_helpers import FLUX, PREC, max_rel_err, residual_term_scale, torch_cuda

pytestmark = pytest.mark.gpu


def _case(ne, p, flux):
    """The first ne tetrahedra of a jittered box in lattice order, all exposed faces walls."""
    m = I.make_box_mesh((3, 2, 2), periodic=(False, False, False), jitter=0.1, shuffle_elements=False)
    vid, xyz, tag = m.tet_vid[:ne], m.tet_xyz[:ne], np.ones((ne, 4), dtype=np.int8)
    P = Problem(vid, xyz, tag, p=p, flux=flux)

    def field(x):
        U = I.entropy_wave(0.4 * x)
        U[..., 3] += 0.1 * x[..., 0]
        return U
    return (vid, xyz, tag), P, P.project(field)


def _mesh(arrays, p, flux, precision):
    return dg.Mesh(*arrays, order=p, precision=PREC[precision], flux=FLUX[flux], renumber=dg.DG_ORDER_MORTON)


@pytest.mark.parametrize("ne", [1, 31, 32, 33, 65])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("precision,flux", [("fp64", "roe"), ("fp32", "roe"), ("fp32", "rusanov")])
def test_rows_at_tile_edges(precision, flux, p, ne):
    torch = torch_cuda()
    arrays, P, U = _case(ne, p, flux)
    M = _mesh(arrays, p, flux, precision)
    Ud = torch.from_numpy(U).cuda()
    out = torch.full_like(Ud, float("nan"))
    dg.dg_residual(M.handle, Ud, out)
    dg.dg_sync_status(M.handle)
    tol, vtol = (1e-12, 1e-11) if precision == "fp64" else (1e-4, 1e-4)
    R = P.residual(U)
    scale = residual_term_scale(P, U)
    assert max_rel_err(out.cpu().numpy(), R, term_scale=scale) < tol
    # one step: dt R enters the state, so its error is dt times the residual's
    dt = P.stable_dt(U, 0.1)
    dg.dg_set_state(M.handle, Ud)
    dg.dg_rk3_step(M.handle, dt, 1)
    dg.dg_get_state(M.handle, out)
    eps = 1e-15 if precision == "fp64" else 6e-7   # rounding of the state itself, a few ulp
    err = np.abs(out.cpu().numpy() - P.rk3_step(U, dt)).max()
    assert err < dt * tol * max(scale) + eps * np.abs(U).max()
    lam = I.random_directions(U.shape, 1)[0]
    dg.dg_residual_vjp(M.handle, Ud, torch.from_numpy(lam).cuda(), out)
    assert max_rel_err(out.cpu().numpy(), P.vjp(U, lam)) < vtol
    M.close()


@pytest.mark.parametrize("flux", ["rusanov", "roe"])
def test_vjp_at_exact_kinks(flux):
    """A stream along x on a lattice of spacing 1/4, where every product of coordinate differences is
    exact: faces parallel to x see a normal velocity of exactly zero, so |u.n| is at its kink, with
    jumps in density and pressure across it; both residuals of such a face take their own interior
    side's branch (the oracle differentiates each by itself)."""
    torch = torch_cuda()
    m = I.make_box_mesh((4, 4, 4), jitter=0.0)
    P = Problem(m.tet_vid, m.tet_xyz, None, p=1, flux=flux)
    U = np.zeros((m.ne, 5, P.nb))
    rho = 1.0 + 0.2 * I.uniform01(11, m.ne)
    U[:, 0, 0], U[:, 1, 0], U[:, 4, 0] = rho, 0.25 * rho, 2.5 + 0.4 * I.uniform01(12, m.ne)
    U /= np.sqrt(6.0)
    lam = I.random_directions(U.shape, 1)[0]
    M = _mesh((m.tet_vid, m.tet_xyz, None), 1, flux, "fp64")
    out = torch.empty(U.shape, dtype=torch.float64, device="cuda")
    dg.dg_residual_vjp(M.handle, torch.from_numpy(U).cuda(), torch.from_numpy(lam).cuda(), out)
    assert max_rel_err(out.cpu().numpy(), P.vjp(U, lam)) < 1e-11
    M.close()
