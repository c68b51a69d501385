"""What the library keeps of the device's memory between calls, in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _run(body):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    code = "import sys\nsys.path.insert(0, '.')\nimport torch\nfrom paper_1810_06760_gb300 import fga, workloads as W\n" + body
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return [float(v) for v in r.stdout.split()]


def test_transform_alone_keeps_little():
    # 860 MB of FP64 scratch for 224^3 points and 192^3 x 3 values; the first call, a small one, loads the kernels
    kept, = _run("""
def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]
descs = []
for ny, nq in ((16, 2), (224, 24)):
    f, y0, dy, mesh, k = W.transform_case(ny=ny, nq=nq)
    f = torch.as_tensor(f, device='cuda')
    descs.append((fga.init_desc(k, f, None, y0, dy, mesh, (0,), fga.PREC_FP64), f))
fga.transform(descs[0][0])
out = torch.empty(((24 * 8,) * 3) + (3,), dtype=torch.complex128, device='cuda')
before = free()
fga.transform(descs[1][0], out=out)
print(before - free())
""")
    assert kept <= (512 << 20) + (16 << 20)


def test_idle_blocks_go_back_on_request_and_the_bound_stays():
    given, refused = _run("""
w = W.smooth(nq=8, np_=6, ny=24, nsteps=8, n_samples=8, rx_side=8, snap_side=0, grid_n=17)
model = fga.model_from_medium(w.medium, 'cuda')
f = torch.as_tensor(w.f, device='cuda')
desc = fga.init_desc(w.k, f, None, w.y0, w.dy, w.mesh, w.classes, fga.PREC_FP32)
solve = lambda: fga.solve(model, desc, w.dt, w.nsteps, w.times, rw=w.rw, rx_axes=w.rx_axes)
u = solve()[0]
fga.set_device_memory_limit(fga.device_memory_in_use() + 2e9)
assert torch.equal(u, solve()[0])
torch.cuda.synchronize()
held = torch.cuda.mem_get_info()[0]
fga.release_idle_memory()
print(torch.cuda.mem_get_info()[0] - held)
assert torch.equal(u, solve()[0])
big = W.smooth(nq=16, np_=8, ny=24, nsteps=8, n_samples=8, rx_side=8, snap_side=0, grid_n=17)   # 1.6 GB of beams, twice
try:
    fga.solve(model, fga.init_desc(big.k, f, None, w.y0, w.dy, big.mesh, big.classes, fga.PREC_FP32), w.dt, w.nsteps,
              w.times, rw=w.rw, rx_axes=w.rx_axes)
    print(0)
except fga.FGAError as e:
    print(1 if e.status == fga.FGA_ERR_OOM else -1)
""")
    # the beam set and its sorted copy alone are 2 x 196 B x 442,368 beams = 173 MB
    assert given > 150e6 and refused == 1
