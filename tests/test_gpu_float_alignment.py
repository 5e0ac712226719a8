"""phi0, phi_out and the outputs of rsf_init_phi0 in device memory at addresses that no float may be
read or written at: such buffers are copied, as host buffers are, and the results are the bits of
aligned ones."""
import ctypes

import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPE = (12, 14, 36)
N = 12 * 14 * 36


def _params(sigma):
    return dict(sigma=sigma, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)


def _inputs():
    rng = np.random.default_rng(4)
    vol = torch.from_numpy(np.rint(rng.uniform(0, 255, size=SHAPE)).astype(np.uint8)).cuda()
    return vol, torch.from_numpy(rng.normal(0.0, 2.0, size=SHAPE).astype(np.float32)).cuda()


def _bytes_at(a, off):
    """a's bytes at `off` past an aligned address, and that buffer."""
    buf = torch.zeros(off + 4 * N, dtype=torch.uint8, device="cuda")
    if a is not None:
        buf[off:] = a.reshape(-1).view(torch.uint8)
    return buf


def _floats(buf, off):
    return buf[off:].cpu().numpy().tobytes()


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    c = rsf.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("off0,off1", [(1, 0), (0, 2), (3, 1)])
@pytest.mark.parametrize("sigma", [3.0, 3.5])
@pytest.mark.parametrize("iters", [1, 3])
def test_evolve(ctx, off0, off1, sigma, iters):
    vol, phi = _inputs()
    ref = ctx.evolve(vol, phi, _params(sigma), iters).cpu().numpy().tobytes()
    src, dst = _bytes_at(phi, off0), _bytes_at(None, off1)
    torch.cuda.synchronize()
    nz, ny, nx = SHAPE
    p = rsf.Params.of(_params(sigma)).tuple()
    st = rsf.load_library().rsf_evolve(ctx.handle, vol.data_ptr(), rsf.RSF_U8, nx, ny, nz, src.data_ptr() + off0,
                                       dst.data_ptr() + off1, *p, iters)
    assert st == 0 and _floats(dst, off1) == ref


@pytest.mark.parametrize("off0,off1", [(1, 2), (2, 0)])
def test_batch_and_serving(ctx, off0, off1):
    vol, phi = _inputs()
    ref = ctx.evolve(vol, phi, _params(3.0), 4).cpu().numpy().tobytes()
    nz, ny, nx = SHAPE
    p = rsf.Params.of(_params(3.0)).tuple()
    L = rsf.load_library()
    src, dst = _bytes_at(phi, off0), _bytes_at(None, off1)
    torch.cuda.synchronize()
    args = (vol.data_ptr(), rsf.RSF_U8, nx, ny, nz, src.data_ptr() + off0, dst.data_ptr() + off1, *p, 4)
    arr = (rsf.Brick * 1)(rsf.Brick(*args))
    assert L.rsf_evolve_batch(ctx.handle, arr, 1) == 0
    assert _floats(dst, off1) == ref
    dst.zero_()
    torch.cuda.synchronize()
    r, t = rsf.Request(*args, rsf.STORAGE["f32"], -1, 0), ctypes.c_uint64()
    served = rsf.Context(0)
    assert L.rsf_submit(served.handle, ctypes.byref(r), ctypes.byref(t)) == 0
    assert L.rsf_wait(served.handle, t, 60000) == 0
    served.close()
    assert _floats(dst, off1) == ref


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("phi_off", [0, 1])
def test_init_outputs(ctx, off, phi_off):
    rng = np.random.default_rng(7)
    vol = rng.normal(0.0, 1.0, size=SHAPE).astype(np.float32)
    vol[5, 5:8, 20:23] += 60.0
    vol = torch.from_numpy(vol).cuda()
    seeds = torch.zeros(SHAPE, dtype=torch.uint8, device="cuda")
    resp = torch.empty(SHAPE, dtype=torch.float32, device="cuda")
    phi, n = ctx.init_phi0(vol, 1.5, 0.3, 2.0, seeds=seeds, response=resp)
    dst, out, mask = _bytes_at(None, off), _bytes_at(None, phi_off), torch.zeros(N + 1, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    nz, ny, nx = SHAPE
    k = ctypes.c_int64()
    st = rsf.load_library().rsf_init_phi0(ctx.handle, vol.data_ptr(), rsf.RSF_F32, nx, ny, nz, 1.5, 0.3, 2.0,
                                          out.data_ptr() + phi_off, ctypes.byref(k), mask.data_ptr() + 1, dst.data_ptr() + off)
    assert st == 0 and k.value == n > 0
    assert _floats(dst, off) == resp.cpu().numpy().tobytes() and _floats(out, phi_off) == phi.cpu().numpy().tobytes()
    assert mask[1:].cpu().numpy().tobytes() == seeds.cpu().numpy().tobytes()
