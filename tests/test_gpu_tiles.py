"""The tiled kernels at the edges of their tiles: one row or column more and less than the x/y
tiles (32 x 48, 40 or 32) and the update's (32 x 14, 12, 10 or 8), odd and even rows, image rows
that the copies read in place and rows that are staged, a few planes and chunks split over
several CTAs; one iteration from a rough phi against the FP64 oracle within the per-step bound.

The exact arithmetic (widths without fast kernels, the forced path, rsf_evolve_noalloc) runs in
the tiled schedule where its fields fit and in the separable passes elsewhere: both give the
same bits."""
import numpy as np
import pytest

import oracle
from paper_2404_02813_gb300 import rsf

from _parity import assert_phi_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")


def _case(shape, dtype, seed):
    rng = np.random.default_rng(seed)
    vol = rng.uniform(0, 255, size=shape)
    vol = vol.astype(np.float32) if dtype == np.float32 else np.rint(vol).astype(dtype)
    phi = (rng.normal(0.0, 2.0, size=shape)).astype(np.float32)
    return vol, phi


def _params(sigma):
    return dict(sigma=sigma, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)


@pytest.mark.parametrize("sigma", [1.0, 1.5, 3.0, 4.0, 5.0, 6.0])
@pytest.mark.parametrize("shape,dtype", [
    ((5, 14, 32), np.uint8), ((9, 15, 33), np.uint16), ((6, 13, 31), np.float32), ((21, 49, 34), np.uint8),
    ((4, 41, 64), np.uint16), ((11, 29, 48), np.float32), ((35, 12, 4), np.uint8)])
@pytest.mark.parametrize("force", ["li", "eq15"])
def test_tile_edges(shape, dtype, sigma, force):
    _gpu()
    vol, phi = _case(shape, dtype, 11)
    p = _params(sigma)
    ctx = rsf.Context(0)
    ctx.set_force(force)
    v, ph = torch.from_numpy(vol).cuda(), torch.from_numpy(phi).cuda()
    ref = oracle.step(vol.astype(np.float64), phi.astype(np.float64), p, **({"force": "eq15"} if force == "eq15" else {}))
    out = ctx.evolve(v, ph, p, 1).cpu().numpy()
    assert_phi_close(out, ref, phi, what=f"{shape} sigma {sigma} {force}")
    ctx.set_option(rsf.OPT_ZCHUNK, 8)  # chunks of their own CTAs
    assert_phi_close(ctx.evolve(v, ph, p, 1).cpu().numpy(), ref, phi, what="z chunks of 8")
    ctx.close()


@pytest.mark.parametrize("sigma", [0.5, 2.5, 3.5, 4.5, 5.5, 6.5, 8.0])
@pytest.mark.parametrize("shape,dtype", [((61, 33, 40), np.uint8), ((240, 217, 5), np.uint16), ((23, 40, 37), np.float32)])
def test_exact_arithmetic_same_bits_tiled_and_in_passes(shape, dtype, sigma):
    """rsf_evolve takes the tiled schedule for each of these; rsf_evolve_noalloc does for the
    first and third and the passes for the second (rows of 5 at a pitch of 32 do not fit)."""
    _gpu()
    vol, phi = _case(shape, dtype, 5)
    p = _params(sigma)
    ctx = rsf.Context(0)
    ctx.set_path("passes")
    v, ph = torch.from_numpy(vol).cuda(), torch.from_numpy(phi).cuda()
    ref = ctx.evolve(v, ph, p, 3).cpu().numpy()
    out = torch.full_like(ph, float("nan"))
    rsf.evolve_noalloc(v, ph, p, 3, out)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), ref)
    # a phi_out of 4-byte alignment only
    buf = torch.full((ph.numel() + 1,), float("nan"), device="cuda")
    odd = buf[1:].view(ph.shape)
    rsf.evolve_noalloc(v, ph, p, 2, odd)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(odd.cpu().numpy(), ctx.evolve(v, ph, p, 2).cpu().numpy())
    one = oracle.step(vol.astype(np.float64), phi.astype(np.float64), p)
    assert_phi_close(ctx.evolve(v, ph, p, 1).cpu().numpy(), one, phi, what=f"{shape} sigma {sigma}")
    ctx.close()
