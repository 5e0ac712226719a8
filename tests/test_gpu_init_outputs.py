"""rsf_init_phi0 with outputs that share memory: the response is written first, then the seed mask,
then phi0, wherever they lie."""
import ctypes

import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (3, 40, 44)
N = 3 * 40 * 44


def _volume():
    rng = np.random.default_rng(7)
    vol = rng.normal(0.0, 1.0, size=SHAPE).astype(np.float32)
    vol[1, 10:13, 20:23] += 60.0
    vol[2, 30:33, 5:8] += 60.0
    return torch.from_numpy(vol).cuda()


def _init(ctx, vol, phi, seeds, resp):
    """Device addresses in, number of seeds out."""
    n = ctypes.c_int64()
    nz, ny, nx = SHAPE
    st = rsf.load_library().rsf_init_phi0(ctx.handle, vol.data_ptr(), rsf.RSF_F32, nx, ny, nz, 1.5, 0.3, 2.0, phi,
                                          ctypes.byref(n), seeds, resp)
    assert st == 0, rsf.load_library().rsf_last_error()
    return int(n.value)


# offsets in bytes of phi0, the mask and the response in one buffer
@pytest.mark.parametrize("at", [(4 * N, 8 * N, 0), (0, 4 * N, 0), (0, N, 4 * N), (0, 0, 0), (2 * N, 3 * N, 0),
                                (4 * N, 2 * N, 0), (2 * N, 5 * N, 3 * N)])
def test_order_of_shared_outputs(at):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    vol = _volume()
    ctx = rsf.Context(0)
    seeds = torch.zeros(SHAPE, dtype=torch.uint8, device="cuda")
    resp = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    phi, n = ctx.init_phi0(vol, 1.5, 0.3, 2.0, seeds=seeds, response=resp)
    assert n > 0
    want = np.zeros(10 * N, dtype=np.uint8)
    for off, a in ((at[2], resp), (at[1], seeds), (at[0], phi)):
        b = a.cpu().numpy().view(np.uint8).reshape(-1)
        want[off:off + b.size] = b
    buf = torch.zeros(10 * N, dtype=torch.uint8, device="cuda")
    base = buf.data_ptr()
    torch.cuda.synchronize()
    assert _init(ctx, vol, base + at[0], base + at[1], base + at[2]) == n
    np.testing.assert_array_equal(buf.cpu().numpy(), want)
    ctx.close()
