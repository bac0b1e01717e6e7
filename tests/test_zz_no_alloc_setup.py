"""The one-time set-up of tc_to_physical_noalloc: the first call on a device is
enough before a stream capture, whatever size it had, and a later one takes no
device memory (a fresh process, because the set-up belongs to the process).  Pairs of a first size and a captured one on
both routes: planned lengths of two and three passes, and unplanned ones."""
import os
import subprocess
import sys

import pytest

from helpers import ensure_lib

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PROGRAM = r"""
import sys
sys.path.insert(0, %r)
import numpy as np, torch
import paper_0711_1429_gb300 as tc
a, b = eval(sys.argv[1]), eval(sys.argv[2])
torch.cuda.init()
def buffers(Nr, Nt, Nz):
    rng = np.random.default_rng(1)
    F = rng.standard_normal((Nr, Nz, Nt // 2)) + 1j * rng.standard_normal((Nr, Nz, Nt // 2))
    return torch.from_numpy(F).cuda(), torch.zeros(Nr * Nz * 3 // 2 * Nt * 3 // 2, dtype=torch.float64, device="cuda")
def call(c, x, out, s):
    tc.tc_to_physical_noalloc(*c, x.data_ptr(), out.data_ptr(), s.cuda_stream)
s = torch.cuda.Stream()
xa, oa = buffers(*a)
xb, ob = buffers(*b)
# torch's own kernels that are used below
z = torch.isfinite(ob).all().item(); ob.zero_(); keep = ob.clone()
torch.cuda.synchronize()
call(a, xa, oa, s)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
if sys.argv[3] == "memory":                    # nothing is loaded or allocated any more
    call(b, xb, ob, s)
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free, free - torch.cuda.mem_get_info()[0]
else:
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="global"):
        call(b, xb, ob, torch.cuda.current_stream())
    g.replay()
    torch.cuda.synchronize()
    graph = ob.clone()
    ob.zero_()
    call(b, xb, ob, s)
    torch.cuda.synchronize()
    assert torch.equal(graph, ob) and bool((ob != 0).any())
print("ok")
"""


@pytest.mark.parametrize("first, second", [((2, 8, 8), (3, 512, 512)), ((2, 512, 512), (3, 1024, 256)),
                                           ((2, 16, 34), (3, 96, 48)), ((3, 96, 48), (2, 16, 34)), ((2, 36, 10), (3, 768, 8))])
@pytest.mark.parametrize("what", ["memory", "capture"])
def test_first_call_of_one_size_sets_up_every_other(first, second, what):
    pytest.importorskip("torch")
    ensure_lib()
    p = subprocess.run([sys.executable, "-c", PROGRAM % ROOT, repr(first), repr(second), what], capture_output=True, text=True, timeout=300)
    assert p.returncode == 0 and p.stdout.strip().endswith("ok"), p.stderr[-2000:]
