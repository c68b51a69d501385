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
