"""Bricks thinner along y than the x/y kernels' tiles (48, 40 or 32 rows), which stage their own rows
and halo alone, and those just not: one iteration from a rough phi against the FP64 oracle within
the per-step bound, alone and in a batch beside a thick brick; the exact arithmetic against the
six passes."""
import numpy as np
import pytest

import oracle
from paper_2404_02813_gb300 import rsf

from _parity import assert_phi_close

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROWS = (4, 5, 31, 32, 33, 39, 40, 41, 47, 48, 49)


def _case(shape, dtype, seed):
    rng = np.random.default_rng(seed)
    vol = rng.uniform(0, 255, size=shape)
    vol = vol.astype(np.float32) if dtype == np.float32 else np.rint(vol).astype(dtype)
    return vol, rng.normal(0.0, 2.0, size=shape).astype(np.float32)


def _params(sigma):
    return dict(sigma=sigma, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)


@pytest.mark.parametrize("sigma", [1.0, 4.0, 6.0])
@pytest.mark.parametrize("force", ["li", "eq15"])
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_one_iteration(sigma, force, dtype):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    ctx = rsf.Context(0)
    ctx.set_force(force)
    items, refs = [], []
    for ny in ROWS:
        vol, phi = _case((6, ny, 35), dtype, ny)
        v, ph = torch.from_numpy(vol).cuda(), torch.from_numpy(phi).cuda()
        ref = oracle.step(vol.astype(np.float64), phi.astype(np.float64), _params(sigma),
                          **({"force": "eq15"} if force == "eq15" else {}))
        out = ctx.evolve(v, ph, _params(sigma), 1).cpu().numpy()
        assert_phi_close(out, ref, phi, what=f"{ny} rows, sigma {sigma}, {force}")
        items.append((v, ph, _params(sigma), 1))
        refs.append(out)
    for o, r in zip(ctx.evolve_batch(items), refs):
        np.testing.assert_array_equal(o.cpu().numpy(), r)
    ctx.close()


@pytest.mark.parametrize("sigma", [3.5, 4.5, 6.5, 8.0])
def test_exact_arithmetic(sigma):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    ctx, passes = rsf.Context(0), rsf.Context(0)
    passes.set_path("passes")
    for ny in ROWS:
        vol, phi = _case((6, ny, 35), np.uint16, ny)
        v, ph = torch.from_numpy(vol).cuda(), torch.from_numpy(phi).cuda()
        np.testing.assert_array_equal(ctx.evolve(v, ph, _params(sigma), 2).cpu().numpy(),
                                      passes.evolve(v, ph, _params(sigma), 2).cpu().numpy(), err_msg=f"{ny} rows")
    ctx.close()
    passes.close()
