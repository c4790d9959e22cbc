"""dg_set_state and dg_get_state convert on the integer pipe and move two values at a time: every kind of
FP64 value, and caller's arrays that are aligned to 8 bytes only, in each storage format.  Expected
values: the conversions' definitions in numpy (FP32 meshes fl32(x); the mixed forms hi = fl32(x),
lo = fl32(x - hi), read back as hi + lo), bitwise but for the payload of a NaN."""
import numpy as np
import pytest

from paper_2209_01877_gb300 import dg
from paper_2209_01877_gb300 import inputs as I

from gpu_helpers import PREC, torch_cuda

pytestmark = pytest.mark.gpu


def _values(n):
    """n FP64 values: exponents over the whole range, around the limits of FP32's normal and subnormal
    numbers and of the integer path (2^-74, 2^126), ties and carries of the 29 dropped bits, special values."""
    rng = np.random.default_rng(3)
    e = np.concatenate([rng.integers(0, 2048, n // 2), 1023 + rng.integers(-160, -60, n // 8),
                        1023 + rng.integers(120, 132, n // 8), 1023 + rng.integers(-20, 20, n - n // 2 - 2 * (n // 8))])
    low = rng.integers(0, 1 << 29, n)
    pick = rng.integers(0, 6, n)
    low = np.where(pick == 0, 0, np.where(pick == 1, 1 << 28, np.where(pick == 2, (1 << 29) - 1, low)))
    high = np.where(rng.integers(0, 4, n) == 0, (1 << 23) - 1, rng.integers(0, 1 << 23, n))
    bits = (rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e.astype(np.uint64) << np.uint64(52)) | \
        (high.astype(np.uint64) << np.uint64(29)) | low.astype(np.uint64)
    x = bits.view(np.float64)
    special = [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 2.0 ** -149, 2.0 ** -126, 2.0 ** -74, 2.0 ** 126, 2.0 ** 128]
    x[:len(special)] = special
    return x


def _expected(x, precision):
    if precision == "fp64":
        return x
    with np.errstate(all="ignore"):
        hi = x.astype(np.float32).astype(np.float64)
        return hi if precision == "fp32" else hi + (x - hi).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("precision", ["fp64", "fp32", "mixed"])
@pytest.mark.parametrize("p", [1, 2, 3])
@pytest.mark.parametrize("dims", [(5, 5, 5), (13, 12, 11)])   # blocks of 8 and of 32 elements, ragged
@pytest.mark.parametrize("offset", [0, 1])                    # 1: the array starts 8 bytes past a 16-byte boundary
def test_state_copies(offset, dims, p, precision):
    torch = torch_cuda()
    m = I.make_box_mesh(dims, jitter=0.1)
    M = dg.Mesh(m.tet_vid, m.tet_xyz, None, order=p, precision=PREC[precision], renumber=dg.DG_ORDER_HILBERT)
    shape = (M.ne, 5, M.nb)
    x = _values(int(np.prod(shape)))
    room = torch.empty(x.size + 2, dtype=torch.float64, device="cuda")
    U = room[offset:offset + x.size].view(shape)
    assert U.data_ptr() % 16 == 8 * offset
    U.copy_(torch.from_numpy(x).view(shape))
    dg.dg_set_state(M.handle, U)
    room.fill_(float("nan"))
    room[0] = room[-1] = 7.0
    if offset == 0:
        room[x.size] = 7.0
    dg.dg_get_state(M.handle, U)
    got, want = U.cpu().numpy().ravel(), _expected(x, precision)
    nan = np.isnan(want)
    np.testing.assert_array_equal(np.isnan(got), nan)
    np.testing.assert_array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
    rest = [0] if offset else [x.size]
    assert all(float(room[i]) == 7.0 for i in rest + [x.size + 1])   # nothing written beside the array
    M.close()
