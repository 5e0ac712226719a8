"""phi0 and phi_out used where the caller has them: the same bits as with host arrays (which are
copied), for one, two and three iterations, with phi_out apart from phi0, the same, shifted over
it by a plane or by one value, or over the volume, and at a 4-byte alignment; phi0 apart from
phi_out stays as it was.  Widths of the fast kernels, of the exact ones and the four-field form."""
import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma,force", [(2.0, "li"), (3.0, "li"), (2.5, "li"), (3.0, "eq15")])
@pytest.mark.parametrize("shape", [(7, 13, 33), (20, 15, 64), (4, 5, 4)])
@pytest.mark.parametrize("iters", [0, 1, 2, 3])
def test_same_bits_where_the_caller_has_it(sigma, force, shape, iters):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    rng = np.random.default_rng(3)
    vol = rng.uniform(0, 255, size=shape).astype(np.float32)
    phi = rng.normal(0.0, 2.0, size=shape).astype(np.float32)
    p = dict(sigma=sigma, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)
    n, plane = phi.size, shape[1] * shape[2]
    ctx = rsf.Context(0)
    ctx.set_force(force)
    ref = ctx.evolve(vol, phi, p, iters, out=np.full_like(phi, np.nan))  # through copies

    def flat(start, size):
        return torch.full((size,), float("nan"), device="cuda")[start:]

    for at, to in ((0, None), (0, 0), (0, plane), (plane, 0), (0, 1), (1, 0), (1, None), (1, 1)):
        buf = flat(0, n + plane + 1)
        src = buf[at:at + n].view(shape)
        src.copy_(torch.from_numpy(phi))
        out = flat(1, n + 1).view(shape) if to is None else buf[to:to + n].view(shape)
        v = torch.from_numpy(vol).cuda()
        ctx.evolve(v, src, p, iters, out=out)
        np.testing.assert_array_equal(out.cpu().numpy(), ref, err_msg=f"phi0 at {at}, phi_out at {to}")
        if to is None:
            np.testing.assert_array_equal(src.cpu().numpy(), phi)
    v = torch.from_numpy(vol).cuda()  # phi_out over the volume
    ctx.evolve(v, torch.from_numpy(phi).cuda(), p, iters, out=v)
    np.testing.assert_array_equal(v.cpu().numpy(), ref)
    ctx.close()
