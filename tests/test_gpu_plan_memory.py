"""Plans under a limit of device memory (GPU).

cudaMalloc and cudaFree of the library go through a host-side stand-in that
refuses what would pass a limit, as the runtime does; nothing is filled up on the
device.  The line table is optional: whatever the limit, a plan that fits without
it is built, and gives the same operators.
"""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
typedef int (*malloc_t)(void **, size_t);
typedef int (*free_t)(void *);
static struct { void *p; size_t n; } held[4096];
static size_t now, most, limit = (size_t)-1, refused;
void fake_limit(size_t n, size_t refuse) /* at most n bytes, and no piece of `refuse` bytes */
{
    limit = n;
    refused = refuse;
    most = now = 0;
    for (int k = 0; k < 4096; ++k) held[k].p = NULL;
}
size_t fake_most(void) { return most; }
int cudaMalloc(void **p, size_t n)
{
    if (now + n > limit || n == refused) return 2; /* cudaErrorMemoryAllocation */
    int e = ((malloc_t)dlsym(RTLD_NEXT, "cudaMalloc"))(p, n);
    if (e) return e;
    now += n;
    if (now > most) most = now;
    for (int k = 0; k < 4096; ++k)
        if (!held[k].p) { held[k].p = *p; held[k].n = n; break; }
    return 0;
}
int cudaFree(void *p)
{
    for (int k = 0; p && k < 4096; ++k)
        if (held[k].p == p) { now -= held[k].n; held[k].p = NULL; }
    return ((free_t)dlsym(RTLD_NEXT, "cudaFree"))(p);
}
"""

SCRIPT = r"""
import ctypes, numpy as np, torch
import synth
import paper_1607_01650_gb300 as dect
fake = ctypes.CDLL(FAKE_SO)
fake.fake_limit.argtypes, fake.fake_most.restype = [ctypes.c_size_t, ctypes.c_size_t], ctypes.c_size_t
g = synth.tiny_geometry(n=96, nv=40, nb=140, px=1.0, sod=300.0, sdd=600.0)
x, y = torch.rand((2, 96, 96), device="cuda"), torch.empty((2, 40, 140), device="cuda")

def build(limit, refuse=0):
    fake.fake_limit(limit, refuse)
    try:
        plan = dect.Plan(g)
        return plan, fake.fake_most()
    except dect.DectError as e:
        assert "memory" in str(e).lower(), e
        return None, 0
    finally:
        fake.fake_limit(2 ** 40, 0)

plan, full = build(2 ** 40)
want = dect.project(plan, x, y).clone()
# without the line table: its fractions, tiles of 32 x 32 of 4 bytes, are refused
plan, need = build(2 ** 40, 40 * 3 * 5 * 4096)
assert 0 < need < full, (need, full)
assert (dect.project(plan, x, y) - want).norm() <= 1e-6 * want.norm()
for limit in [need + (full - need) * k // 16 for k in range(17)]:
    plan, _ = build(limit)
    assert plan is not None, (limit, need, full)
    assert (dect.project(plan, x, y) - want).norm() <= 1e-6 * want.norm()
plan, _ = build(need - 1)
assert plan is None
print("memory ok")
"""


def test_plan_that_fits_without_the_line_table_is_built(tmp_path):
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-L", CUDA + "/lib64", "-Wl,--no-as-needed",
                    "-lcudart", "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so),
               LD_LIBRARY_PATH=CUDA + "/lib64:" + os.environ.get("LD_LIBRARY_PATH", ""))
    r = subprocess.run([sys.executable, "-c", SCRIPT.replace("FAKE_SO", repr(str(so)))], cwd=ROOT, env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "memory ok" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
