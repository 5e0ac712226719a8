"""RSF_PATH_PASSES runs the six separable passes, whatever the radius: their kernels launch and no
tiled one.  The exact arithmetic of the tiled schedule (the default at the widths without fast
kernels) gives the passes' bits, phi and the stage dump alike, at every radius 1 to 16 that the
default takes there and through rsf_evolve_noalloc at all of them, on volumes of more than one tile
along x and y.  Radius 0 has the passes alone: one iteration against the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2404_02813_gb300 import rsf

from _parity import assert_phi_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TILED_RADII = (2, 3, 4, 5, 6, 8, 10, 12)  # the default path's fast arithmetic


@pytest.fixture(scope="module")
def ctxs():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    default, passes = rsf.Context(0), rsf.Context(0)
    passes.set_path("passes")
    yield default, passes
    default.close()
    passes.close()


def _case(shape, dtype, seed):
    rng = np.random.default_rng(seed)
    vol = rng.uniform(0, 255, size=shape)
    vol = vol.astype(np.float32) if dtype == np.float32 else np.rint(vol).astype(dtype)
    phi = rng.normal(0.0, 2.0, size=shape).astype(np.float32)
    return vol, phi, torch.from_numpy(vol).cuda(), torch.from_numpy(phi).cuda()


def _params(radius):
    return dict(sigma=radius / 2 if radius else 0.2, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0,
                dt=0.1)


@pytest.mark.parametrize("radius", [0, 6, 7])
def test_the_option_runs_the_passes(ctxs, radius):
    _, _, v, ph = _case((9, 20, 40), np.uint8, 1)
    ctx = ctxs[1]
    ctx.prof_enable(True)
    ctx.evolve(v, ph, _params(radius), 2)
    ran = {k for k, (n, _) in ctx.prof_get().items() if n}
    ctx.prof_enable(False)
    assert ran and not any(k.startswith(("rsf_ta", "rsf_tb")) for k in ran), ran


@pytest.mark.parametrize("radius", range(1, 17))
@pytest.mark.parametrize("shape,dtype", [((37, 35, 34), np.uint8), ((9, 53, 70), np.uint16), ((23, 40, 37), np.float32)])
def test_exact_tiled_bits_at_every_radius(ctxs, shape, dtype, radius):
    _, _, v, ph = _case(shape, dtype, 5)
    p = _params(radius)
    ref = ctxs[1].evolve(v, ph, p, 3)
    out = torch.full_like(ph, float("nan"))
    rsf.evolve_noalloc(v, ph, p, 3, out)  # the tiled schedule: these volumes' fields fit its memory
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.cpu().numpy(), ref.cpu().numpy())
    if radius not in TILED_RADII:
        np.testing.assert_array_equal(ctxs[0].evolve(v, ph, p, 3).cpu().numpy(), ref.cpu().numpy())
        a, b = ctxs[0].step_stages(v, ph, p), ctxs[1].step_stages(v, ph, p)
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())


@pytest.mark.parametrize("shape,dtype", [((9, 20, 40), np.uint8), ((12, 7, 33), np.float32)])
@pytest.mark.parametrize("poison", [0, 1])
def test_radius_0_against_the_oracle(shape, dtype, poison):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    vol, phi, v, ph = _case(shape, dtype, 2)
    p = _params(0)
    ctx = rsf.Context(0)
    ctx.set_option(rsf.OPT_POISON, poison)
    ref, d = oracle.step(vol.astype(np.float64), phi.astype(np.float64), p, dump=True)
    out, st = ctx.step_stages(v, ph, p)
    assert_phi_close(out.cpu().numpy(), ref, phi, what=f"{shape} radius 0")
    np.testing.assert_allclose(st[4].cpu().numpy(), d["lap"], atol=1e-4, rtol=0)
    np.testing.assert_array_equal(ctx.evolve(v, ph, p, 1).cpu().numpy(), out.cpu().numpy())
    ctx.close()
