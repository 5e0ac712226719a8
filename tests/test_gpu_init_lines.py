"""The seed initialisation's kernels at their edges: lines shorter and longer than a group of
8, at the switch from 32 to 8 columns per block, ragged tiles, every radius with a kernel of
its own and radii without.  Squared distances are exact integers and the square root and
subtraction are correctly rounded, so phi0 is compared bit for bit; the response within the
bound of test_gpu_init (FP32 filters)."""
import numpy as np
import pytest

import oracle
from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
ndi = pytest.importorskip("scipy.ndimage")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,s", [
    ((1, 4, 4), 0.4), ((3, 9, 33), 0.7), ((8, 31, 65), 1.0), ((9, 64, 32), 1.5), ((17, 70, 40), 2.0),
    ((2, 45, 100), 3.0), ((5, 33, 37), 5.3), ((1, 1430, 40), 1.5), ((2, 1700, 9), 1.0), ((1500, 5, 12), 1.0),
    ((7, 4, 2100), 2.0)])
def test_lines_and_radii(shape, s):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    rng = np.random.default_rng(7)
    vol = rng.normal(0.0, 1.0, size=shape).astype(np.float32)
    for _ in range(3):  # a few bright blobs, so that seeds are sparse
        c = [int(rng.integers(n)) for n in shape]
        vol[tuple(slice(max(0, k - 1), k + 2) for k in c)] += 60.0
    seeds = torch.zeros(shape, dtype=torch.uint8, device="cuda")
    resp = torch.empty(shape, dtype=torch.float32, device="cuda")
    ctx = rsf.Context(0)
    phi, n = ctx.init_phi0(torch.from_numpy(vol).cuda(), s, 0.3, 2.0, seeds=seeds, response=resp)
    ctx.close()
    seeds, resp, phi = seeds.cpu().numpy().astype(bool), resp.cpu().numpy(), phi.cpu().numpy()
    assert n == int(seeds.sum()) > 0
    np.testing.assert_array_equal(seeds, oracle.seeds_from_response(resp.astype(np.float64), 0.3))
    ref = oracle.doh_response(vol.astype(np.float64), s)
    fin = np.isfinite(ref) & np.isfinite(resp)
    np.testing.assert_allclose(resp[fin], ref[fin], rtol=0, atol=2e-5 * np.abs(ref[fin]).max())
    d2 = np.rint(ndi.distance_transform_edt(~seeds) ** 2).astype(np.float32)
    np.testing.assert_array_equal(phi, np.float32(2.0) - np.sqrt(d2))
