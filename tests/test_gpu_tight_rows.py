"""The Eq. (15) form with a 16-bit storage option on images whose rows need a padded copy: batched
and served bricks, where the copy shares the q and stage blocks, give rsf_evolve's bits (its blocks
are larger), also with every field poisoned before the first iteration."""
import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [np.uint8, np.uint16, np.float32])
@pytest.mark.parametrize("nx", [4, 5, 9, 29, 30, 31, 32, 33, 65, 127, 253])
def test_copied_image_shares_the_blocks(dtype, nx):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (6, 11, nx)
    rng = np.random.default_rng(nx)
    vol = torch.from_numpy(rng.integers(0, 256, size=shape).astype(dtype)).cuda()
    phi = torch.from_numpy(rng.normal(0.0, 2.0, size=shape).astype(np.float32)).cuda()
    p = dict(sigma=2.0, eps=1.0, lambda1=0.1, lambda2=0.1, nu=58.5, mu=1.0, dt=0.06)
    ctx = rsf.Context(0)
    ctx.set_force("eq15")
    ref = ctx.evolve(vol, phi, p, 3).cpu().numpy()
    ctx.set_storage("f16")
    ctx.set_option(rsf.OPT_POISON, 1)
    for out in ctx.evolve_batch([(vol, phi, p, 3)] * 3):
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
    out = torch.empty_like(phi)
    ctx.wait(ctx.submit(vol, phi, p, 3, out, storage="f16"))
    np.testing.assert_array_equal(out.cpu().numpy(), ref)
    ctx.close()
