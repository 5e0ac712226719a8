"""rsf_init_phi0 with outputs that share memory: the response is written first, then the seed mask,
then phi0, wherever they lie.  The response at every filter radius."""
import ctypes

import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("radius", range(17))
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_response_at_every_radius(radius, dtype):
    """Ragged tiles; the bound of test_gpu_init_lines (FP32 filters)."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    rng = np.random.default_rng(radius)
    vol = rng.uniform(0.0, 60.0, size=(2, 45, 71))
    vol[1, 20:23, 30:33] += 150.0
    vol = np.rint(vol).astype(dtype)
    s = radius / 3 if radius else 0.1
    resp = torch.empty(vol.shape, dtype=torch.float32, device="cuda")
    ctx = rsf.Context(0)
    ctx.init_phi0(torch.from_numpy(vol).cuda(), s, 0.3, 2.0, response=resp)
    ctx.close()
    resp, ref = resp.cpu().numpy(), oracle.doh_response(vol.astype(np.float64), s)
    fin = np.isfinite(ref) & np.isfinite(resp)
    assert fin.any()
    np.testing.assert_allclose(resp[fin], ref[fin], rtol=0, atol=2e-5 * np.abs(ref[fin]).max())
