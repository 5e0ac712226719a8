"""Calls whose working memory fills the context's budget to the byte: each path takes no more than
the fields it documents, so that descriptors and tables of its own never turn such a call away."""
import numpy as np
import pytest

from paper_2404_02813_gb300 import rsf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

STATS = 4 * 3 * 1024           # partial sums of the image statistics
LANE = 16 * 1024 + 4 * 4 * 32  # launch descriptors of one serving lane (16 bricks)


def _align(b):
    return (b + 255) // 256 * 256


def _params(sigma):
    return dict(sigma=sigma, eps=1.0, lambda1=1.0, lambda2=2.0, nu=0.004 * 255.0 ** 2, mu=1.0, dt=0.1)


def _case(shape, seed=4):
    rng = np.random.default_rng(seed)
    v = torch.from_numpy(np.rint(rng.uniform(0, 255, size=shape)).astype(np.uint8)).cuda()
    return v, torch.from_numpy(rng.normal(0.0, 2.0, size=shape).astype(np.float32)).cuda()


def _voxels(shape):
    nz, ny, nx = shape
    return nx * ny * nz, (nx + 31) // 32 * 32 * ny * nz


def _brick(shape):
    """phi, its copy and the q block; profiles; constants; the FP32 stage block."""
    n, np_ = _voxels(shape)
    return 4 * _align(4 * n) + _align(4 * sum(shape)) + 256 + _align(28 * np_)


@pytest.mark.parametrize("sigma", [0.5, 3.5])
@pytest.mark.parametrize("shape", [(4, 4, 4), (20, 18, 37)])
def test_evolve_at_a_width_without_fast_kernels(sigma, shape):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    v, ph = _case(shape)
    n, np_ = _voxels(shape)
    free = rsf.Context(0)
    ref = free.evolve(v, ph, _params(sigma), 2).cpu().numpy()
    free.close()
    tight = rsf.Context(0, 5 * 4 * n + 8 * 4 * np_ + 4 * sum(shape) + 16 + STATS)
    np.testing.assert_array_equal(tight.evolve(v, ph, _params(sigma), 2).cpu().numpy(), ref)
    tight.close()


def test_many_bricks_without_iterations():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape, nb = (4, 4, 4), 200
    v, ph = _case(shape)
    ctx = rsf.Context(0, nb * _brick(shape) + STATS)
    for out in ctx.evolve_batch([(v, ph, _params(3.0), 0)] * nb):
        np.testing.assert_array_equal(out.cpu().numpy(), ph.cpu().numpy())
    ctx.close()


def test_curtain_of_many_subvolumes():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape, edge, curtain = (4, 4, 20000), 4, 2
    v, ph = _case(shape)
    nb = (shape[2] - edge + 1) // 2 + 1
    sub = _align(edge ** 3) + _align(4 * edge ** 3)
    tables = 8 * nb + 4 * (nb + 2) + sum(4 * n * (1 + 2 * 4) + 4 * n * 4 for n in shape)
    ctx = rsf.Context(0, nb * (sub + _brick((edge,) * 3)) + _align(tables) + 1024 + STATS)
    out = ctx.evolve_curtain(v, ph, _params(3.0), 0, edge, curtain)
    np.testing.assert_allclose(out.cpu().numpy(), ph.cpu().numpy(), rtol=2.0 ** -22, atol=0)
    ctx.close()


def test_served_requests_of_two_groups():
    """Two requests of one size class and different widths, budgeted with the descriptors of one lane."""
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    shape = (20, 24, 32)
    v, ph = _case(shape)
    ctx = rsf.Context(0, 2 * _brick(shape) + STATS + LANE)
    ref = rsf.Context(0)
    outs = [torch.full_like(ph, float("nan")) for _ in range(2)]
    tickets = [ctx.submit(v, ph, _params(s), 40, o) for s, o in zip((2.0, 3.0), outs)]
    for t in tickets:
        assert ctx.wait(t, 60000) == 0
    for s, o in zip((2.0, 3.0), outs):
        np.testing.assert_array_equal(o.cpu().numpy(), ref.evolve(v, ph, _params(s), 40).cpu().numpy())
    ctx.close()
    ref.close()
