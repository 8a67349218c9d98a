"""What the FP64 mode does where device memory for its digit tables or tiles is not to be had: a cudaMalloc of the test's
own, preloaded into a process of its own, refuses requests above a limit."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
int cudaMalloc(void **p, size_t n)
{
    static int (*real)(void **, size_t);
    if (!real) real = (int (*)(void **, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    if (!real) real = (int (*)(void **, size_t))dlsym(dlopen("libcudart.so.13", RTLD_NOW), "cudaMalloc");
    const char *s = getenv("REFUSE_ABOVE");
    return s && n > strtoull(s, 0, 10) ? 2 : real(p, n);   /* cudaErrorMemoryAllocation */
}
"""

SCRIPT = r"""
import os
import torch
import test_gpu_digits as d
import paper_2501_17967_gb300 as bc

tree, x = d.make(9, 30)
torch.cuda.synchronize()
os.environ["REFUSE_ABOVE"] = "{limit}"
if "{what}" == "tables":
    tree, x = d.make(9, 30)
u, h = d.digits(tree, x, False), d.digits(tree, x, True)
if "{what}" == "tiles":
    assert "FP64 kernels" in bc._load().bc_last_error().decode()
assert torch.equal(u, d.kernels(tree, x, False)) and torch.equal(h, d.kernels(tree, x, True))
del os.environ["REFUSE_ABOVE"]
tree, x = d.make(9, 30)
u = d.digits(tree, x, False)
assert not torch.equal(u, d.kernels(tree, x, False)) and d.relerr(u, d.kernels(tree, x, False)) <= d.BAR
print("served")
"""


# p = 9, some 700 leaves: the digit tables are above 50 MB in one request, a tree's tiles above 10; all else below 3
@pytest.mark.parametrize("what,limit", [("tables", 20_000_000), ("tiles", 3_000_000)])
def test_fp64_without_memory_for_the_digits(what, limit, tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, lib = tmp_path / "refuse.c", tmp_path / "refuse.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    env.pop("REFUSE_ABOVE", None)
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(what=what, limit=limit)], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and "served" in r.stdout, r.stdout + r.stderr
