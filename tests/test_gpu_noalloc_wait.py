"""rsf_evolve_noalloc when a kernel's bounded wait runs out: phi_out is NaN throughout, whether the
last iteration wrote it or the static array; the next call on the device is unaffected.  Driven
without a fault: the copy barriers expect 16 bytes more than arrive, every wait gives up."""
import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("iters", [1, 2])
def test_expired_wait_gives_nan(iters):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (17, 16, 33)
    nz, ny, nx = shape
    rng = np.random.default_rng(4)
    vol = torch.from_numpy(np.rint(rng.uniform(0, 255, size=shape)).astype(np.uint8)).cuda()
    phi = torch.from_numpy(rng.normal(0.0, 2.0, size=shape).astype(np.float32)).cuda()
    p = dict(sigma=2.0, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)
    ref, out = torch.empty_like(phi), torch.zeros_like(phi)
    rsf.evolve_noalloc(vol, phi, p, iters, ref)  # leaves plausible fields in the static array
    torch.cuda.synchronize()
    f = rsf.load_library().rsf_test_noalloc_expired_waits
    f.argtypes = rsf.load_library().rsf_evolve_noalloc.argtypes
    st = f(vol.data_ptr(), rsf.RSF_U8, nx, ny, nz, phi.data_ptr(), out.data_ptr(), *rsf.Params.of(p).tuple(), iters,
           torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert st == 0 and bool(torch.isnan(out).all())
    rsf.evolve_noalloc(vol, phi, p, iters, out)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
