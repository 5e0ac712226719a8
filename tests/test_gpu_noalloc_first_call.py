"""The first rsf_evolve_noalloc on a device is the one that loads code and looks addresses up: later
calls take no device memory, at whatever kernel width and image type, and can be captured."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SCRIPT = """
import numpy as np, torch
from paper_2404_02813_gb300 import rsf
shape = (40, 36, 33)
def params(radius):
    return dict(sigma=radius / 2 if radius else 0.2, eps=1.0, lambda1=1.0, lambda2=2.0, nu=260.1, mu=1.0, dt=0.1)
g = torch.Generator().manual_seed(1)
vols = [(torch.rand(shape, generator=g) * 255).to(torch.uint8).cuda(), (torch.rand(shape, generator=g) * 255).cuda()]
vols.append(vols[0].cpu().to(torch.int32).numpy().astype(np.uint16))
vols[2] = torch.from_numpy(vols[2]).cuda()
ph = torch.randn(shape, generator=g).cuda()
out = [torch.empty_like(ph) for _ in range(17)]
thin_shape = (240, 217, 5)
thin_v, thin_ph = torch.zeros(thin_shape, dtype=torch.uint8, device="cuda"), torch.ones(thin_shape, device="cuda")
side = torch.cuda.Stream()
torch.cuda.synchronize()
rsf.evolve_noalloc(vols[0], ph, params(2), 1, out[0], stream=side)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for r in range(17):
    rsf.evolve_noalloc(vols[r % 3], ph, params(r), 2, out[r], stream=side)
rsf.evolve_noalloc(thin_v, thin_ph, params(4), 1, thin_ph, stream=side)
torch.cuda.synchronize()
now = torch.cuda.mem_get_info()[0]
assert now == free, (free, now)
print("ok")
"""

CAPTURE = SCRIPT.split("free = ")[0] + """
graph = torch.cuda.CUDAGraph()
res = torch.empty_like(ph)
with torch.cuda.graph(graph, stream=side):
    rsf.evolve_noalloc(vols[1], ph, params(9), 3, res, stream=side)
graph.replay()
torch.cuda.synchronize()
rsf.evolve_noalloc(vols[1], ph, params(9), 3, out[1], stream=side)
torch.cuda.synchronize()
assert torch.equal(res, out[1])
print("ok")
"""


@pytest.mark.parametrize("script", [SCRIPT, CAPTURE], ids=["memory", "capture"])
def test_later_calls_load_nothing(script):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", script], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
