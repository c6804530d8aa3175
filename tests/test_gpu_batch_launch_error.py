"""A batch whose sweep launch is refused: the launches beside it are still joined
into the batch's stream, so that what follows on it (a read, a destroy) waits for
them.  The refusal is a fake of the launcher that a child process preloads."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static int left = -1;
void fail_sweep_launch(int n) { left = n; }
typedef int fn(int, const void *, const void *, int, unsigned *, int, int, size_t, void *, _Bool);
int launch(int bits, const void *inst, const void *items, int n, unsigned *queue, int grid, int threads, size_t smem,
           void *stream, _Bool prepare) __asm__("%(symbol)s");
int launch(int bits, const void *inst, const void *items, int n, unsigned *queue, int grid, int threads, size_t smem,
           void *stream, _Bool prepare) {
    if (!prepare && left >= 0 && left-- == 0) return 701;  /* cudaErrorLaunchOutOfResources */
    fn *real = (fn *)dlsym(dlopen("%(lib)s", RTLD_NOW | RTLD_NOLOAD), "%(symbol)s");
    return real(bits, inst, items, n, queue, grid, threads, smem, stream, prepare);
}
"""

CHILD = r"""
import ctypes, sys
sys.path.insert(0, %(root)r)
import pytest
from paper_1312_3004_gb300 import Batch
from paper_1312_3004_gb300._lib import RewlError

def job(L, K, seed):
    return dict(q=10, L=L, h=2, overlap=0.75, m=2, lnf_final=1e-6, flatness=0.8, exchange_interval=K, seed=seed)

# three sizes of walker, three launches: the largest first, then the long one, then the refused one
b = Batch([job(64, 10, 1), job(32, 2_000_000, 2), job(8, 10, 3)], lanes=32)
ctypes.CDLL(None).fail_sweep_launch(2)
with pytest.raises(RewlError):
    b.run_async(1)
b.sync()
steps = [int(b.instance(i).get("steps")[0]) for i in range(3)]
assert steps == [10, 2_000_000, 0], steps
b.close()
b = Batch([job(64, 10, 1), job(32, 1000, 2), job(8, 10, 3)], lanes=32)  # and goes on working
b.run(2)
assert [int(b.instance(i).get("steps")[0]) for i in range(3)] == [20, 2000, 20]
print("joined")
"""


def test_a_refused_launch_leaves_no_work_behind(tmp_path):
    from paper_1312_3004_gb300 import build

    lib = build.build()
    names = subprocess.run(["nm", "-D", "--defined-only", lib], capture_output=True, text=True, check=True).stdout.split()
    symbol = next(n for n in names if "launch_batch_sweep" in n)
    src, so = str(tmp_path / "fake.c"), str(tmp_path / "fake.so")
    with open(src, "w") as f:
        f.write(FAKE % {"symbol": symbol, "lib": lib})
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", so, src, "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}], env=dict(os.environ, LD_PRELOAD=so), cwd=ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "joined" in r.stdout, r.stdout[-2000:] + r.stderr[-3000:]
