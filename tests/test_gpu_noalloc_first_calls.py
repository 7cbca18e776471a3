"""ttcross_sampled_error_noalloc, in a process of its own: after a first call (few samples, small
cores) the calls of every other size allocate no device memory and can be captured
in a CUDA graph at once, whichever kernels they run."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
import sys
import torch
from paper_2407_11290_gb300 import ttcross as tt
n = [40, 30, 20, 35]
cores = {s: [torch.rand(a, m, b, dtype=torch.float64, device="cuda") / s
             for a, m, b in zip([1, s, s, s], n, [s, s, s, 1])] for s in (3, 9, 20, 40, 70, 200)}
out = torch.zeros(1, dtype=torch.float64, device="cuda")
side = torch.cuda.Stream()


def call(s, ns, stream=None):
    tt.sampled_error_noalloc(n, {"kind": "hilbert"}, cores[s], ns, 5, out, stream=stream)


call(3, 100)
torch.cuda.synchronize()
sizes = [(3, 100), (9, 20000), (20, 30000), (40, 20000), (70, 20000), (200, 5000)]
free = torch.cuda.mem_get_info()[0]
if sys.argv[1] == "bytes":
    for s, ns in sizes:
        call(s, ns)
        torch.cuda.synchronize()
        assert torch.cuda.mem_get_info()[0] == free, (s, ns, free - torch.cuda.mem_get_info()[0])
else:
    for s, ns in sizes:
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            call(s, ns, side)
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        captured = out.item()
        call(s, ns)
        torch.cuda.synchronize()
        assert captured == out.item() != 0.0, (s, ns)
print("fine")
"""


@pytest.mark.parametrize("what", ["bytes", "capture"])
def test_first_calls_of_other_sizes(what):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", PROGRAM, what], cwd=root, capture_output=True, text=True,
                       timeout=300, env={**os.environ, "PYTHONPATH": root})
    assert r.returncode == 0 and "fine" in r.stdout, r.stderr[-2000:]
