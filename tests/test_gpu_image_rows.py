"""Images that the set-up copies to a pitch: rows of one and several rounds of a warp's loads, rows
that are multiples of four bytes and not, bases at every byte or element offset.  The result has
the bits that the same image gives from the host, where its copy on the device is aligned."""
import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("nx", [4, 18, 36, 127, 128, 132, 258])
def test_copied_rows(dtype, nx):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (5, 9, nx)
    rng = np.random.default_rng(nx)
    vol = rng.integers(0, 256, size=shape).astype(dtype)
    phi = rng.normal(0.0, 2.0, size=shape).astype(np.float32)
    p = dict(sigma=2.0, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)
    ctx = rsf.Context(0)
    ref = ctx.evolve(vol, phi, p, 2)
    for off in range(4):
        buf = torch.zeros(vol.size + 4, dtype=torch.from_numpy(vol).dtype, device="cuda")
        v = buf[off:off + vol.size].view(shape)
        v.copy_(torch.from_numpy(vol))
        out = ctx.evolve(v, torch.from_numpy(phi).cuda(), p, 2).cpu().numpy()
        np.testing.assert_array_equal(out, ref, err_msg=f"{off} elements off")
        outs = ctx.evolve_batch([(v, torch.from_numpy(phi).cuda(), p, 2)] * 2)
        for o in outs:
            np.testing.assert_array_equal(o.cpu().numpy(), ref, err_msg=f"batched, {off} elements off")
    ctx.close()
