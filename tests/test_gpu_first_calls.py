"""First calls on a fresh mesh: what a call sets up on its first use must not keep it from where later
calls may go."""
import numpy as np
import pytest

from paper_2209_01877_gb300 import dg
from paper_2209_01877_gb300 import inputs as I

from gpu_helpers import FLUX, PREC, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,dims", [("fp64", (4, 4, 4)), ("fp32", (4, 4, 4)), ("fp32", (9, 9, 9))])
@pytest.mark.parametrize("call", ["residual_vjp", "rk3_step_vjp"])
def test_first_adjoint_call_may_be_captured(call, precision, dims):
    """The call allocates on its first use (which a relaxed capture permits) and waits for nothing on
    the host; the graph replays to what the call gives outside a capture, bitwise."""
    torch = torch_cuda()
    m = I.make_box_mesh(dims, jitter=0.1)
    make = lambda: dg.Mesh(m.tet_vid, m.tet_xyz, None, order=2, precision=PREC[precision], flux=FLUX["roe"])   # noqa: E731
    M, fresh = make(), make()
    U = torch.from_numpy(M.project(lambda x: I.isentropic_vortex(x, radius=0.2))).cuda()
    lam = torch.from_numpy(I.random_directions(U.shape, 1)[0]).cuda()
    want, got = torch.empty_like(U), torch.full_like(U, float("nan"))

    def run(mesh, out):
        if call == "residual_vjp":
            dg.dg_residual_vjp(mesh.handle, U, lam, out)
        else:
            dg.dg_rk3_step_vjp(mesh.handle, U, 1e-3, lam, out)

    run(M, want)      # also loads the kernels
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        run(fresh, got)
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())
    del g
    M.close()
    fresh.close()
