"""gd_neighbors_fixed allocates nothing on the host either, so no std::bad_alloc can leave its C entry:
a child process counts the calling thread's operator new during a call (a preloaded replacement of it)
and compares the lists with the oracle's.  Sizes of one leaf, of several levels and of the limit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

COUNTER = """
#include <cstdlib>
#include <new>
static thread_local bool counting = false;
static thread_local long calls = 0;
extern "C" void count_start() { calls = 0; counting = true; }
extern "C" long count_stop() { counting = false; return calls; }
void* operator new(std::size_t n) {
  if (counting) ++calls;
  void* p = std::malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

CHILD = """
import ctypes, sys
import numpy as np, torch
from paper_2609_35967_gb300 import binding as gd, workloads as W
from oracle import gdo
count = ctypes.CDLL(sys.argv[1])
count.count_stop.restype = ctypes.c_long
n, K = int(sys.argv[2]), 16
ins = W.patch_instance(n, K=K, seed=12)
params = gd.instance_params(ins["params"])
xs = [torch.as_tensor(ins[k], device="cuda:0") for k in ("x", "y", "z")]
for it in range(2):
    nbr = torch.full((n, K), -7, dtype=torch.int32, device="cuda:0")
    torch.cuda.synchronize()
    args = (xs[0].data_ptr(), xs[1].data_ptr(), xs[2].data_ptr(), n, K, params, nbr.data_ptr(), 0, 0)
    count.count_start()
    gd.gd_neighbors_fixed(*args)
    calls = count.count_stop()
    torch.cuda.synchronize()
idx = np.unique(np.linspace(0, n - 1, 500).astype(np.int64))
ref, _ = gdo.knn(gdo.params(ins["params"]), ins["x"], ins["y"], ins["z"], idx)
assert np.array_equal(nbr.cpu().numpy()[idx], ref)
print("calls", calls)
"""


@pytest.mark.parametrize("n", [20, 3000, 65536])
def test_no_host_allocation(tmp_path, n):
    src, lib = tmp_path / "count.cc", tmp_path / "libcount.so"
    src.write_text(COUNTER)
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", "-o", str(lib), str(src)], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=root)
    run = subprocess.run([sys.executable, "-c", CHILD, str(lib), str(n)], capture_output=True, text=True, env=env,
                         cwd=root, timeout=300)
    assert run.returncode == 0, run.stderr
    assert run.stdout.split() == ["calls", "0"]
