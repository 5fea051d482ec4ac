"""FP32C's first-half slots when device memory runs out (marked gpu): they are
wanted, never needed.  The memory is a fake's: a preloaded cudaMalloc that
refuses what would take the process past a limit the test sets, so that no
device is filled.

* A limit that leaves the slots their full size, one slot per SM or nothing
  (where the run's other buffers just fit): every run is done, with the slots
  that fit, and the energies agree (the slot counts of one kernel bit for bit,
  the kernel without slots at the form's 2e-6 of |E_J|, test_gpu_parity).
* Integrals added, another form run and a doubles iteration begun when the slots
  hold the last of the memory: the slots make room."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_1409_2700_gb300")
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#include <dlfcn.h>
#include <stddef.h>
#define REAL(name) dlsym(dlopen(CUDART, RTLD_LAZY), name)
static size_t limit = (size_t)1 << 62, used;
static void* ptr[4096];
static size_t len[4096];
void shim_limit(size_t n) { limit = n; }
size_t shim_used(void) { return used; }
int cudaMalloc(void** p, size_t n)
{
    static int (*real)(void**, size_t);
    if (!real) real = (int (*)(void**, size_t))REAL("cudaMalloc");
    if (used + n > limit) return 2;                    /* cudaErrorMemoryAllocation */
    const int e = real(p, n);
    for (int k = 0; !e && k < 4096; k++)
        if (!ptr[k]) { ptr[k] = *p; len[k] = n; used += n; break; }
    return e;
}
int cudaFree(void* p)
{
    static int (*real)(void*);
    if (!real) real = (int (*)(void*))REAL("cudaFree");
    for (int k = 0; p && k < 4096; k++)
        if (ptr[k] == p) { ptr[k] = 0; used -= len[k]; break; }
    return real(p);
}
"""

CHILD = r"""
import ctypes, sys
import numpy as np
sys.path[:0] = [sys.argv[1], sys.argv[1] + "/tests"]
import paper_1409_2700_gb300 as M
from helpers import rand_dimer
shim = ctypes.CDLL(sys.argv[2])
shim.shim_used.restype = ctypes.c_size_t
shim.shim_limit.argtypes = [ctypes.c_size_t]
sms = int(sys.argv[3])
used, ANY = shim.shim_used, 400 << 20                  # below the 512 MB chunk integrals are kept in
slots = lambda per_sm: 256 + per_sm * sms * 12 * 4 * 512       # nX * (oY = 4) * 32 rows of 16 bytes
rng = np.random.default_rng(1)
A, K, CX, eX, CY, eY = rand_dimer(rng, 12, 14, 3, 4)
ab = np.concatenate([A.ravel(), K.ravel()])

def context(dimers):
    shim.shim_limit(ANY)
    ctx = M.Context(precision="fp32c")
    for d in range(dimers):
        ctx.add_dimer(ctx.add_monomer(CX, eX, 3), ctx.add_monomer(CY, eY, 4), ab, M.MCPT_AO_BLOCKS)
    return ctx

def run(ctx, limit):
    shim.shim_limit(limit)
    ctx.run()
    return ctx.energies()[2].copy()

def close(a, b):
    return np.all(np.abs(a - b) <= 2e-6 * np.abs(b[:, :1]))

with context(30) as ctx:
    ref = run(ctx, ANY)
    full = used()
with context(30) as ctx:                               # what the run needs without slots
    bare = full - slots(2)
    got = run(ctx, bare)
    assert used() == bare and close(got, ref), (used(), bare)
for room, left in ((slots(2), 2), (slots(2) - 1, 1), (slots(1), 1), (slots(1) - 1, 0), (1, 0)):
    with context(30) as ctx:
        got = run(ctx, bare + room)
        assert used() == bare + (slots(left) if left else 0), (room, left, used() - bare)
        assert np.array_equal(got, ref) if left else close(got, ref)
        assert np.array_equal(run(ctx, bare + room), got)
# integrals added, to the last byte that the slots would take
with context(30) as ctx:
    run(ctx, full)
    more = 0
    try:
        while more < 200:
            ctx.add_dimer(ctx.add_monomer(CX, eX, 3), ctx.add_monomer(CY, eY, 4), ab, M.MCPT_AO_BLOCKS)
            more += 1
    except M.McptError as e:
        assert e.status == M.MCPT_ENOMEM
    block = (ab.nbytes + 255) // 256 * 256
    assert slots(2) // block <= more <= slots(2) // block + 1, more    # the slots' room, and nothing before it
    got = run(ctx, ANY)
    assert np.all(got == got[0]) and np.array_equal(got[0], ref[0])
# another form's run, and the doubles iteration
with context(30) as ctx:
    run(ctx, full)
    ctx.set_precision("fp64")
    got = run(ctx, full)
    assert close(got, ref)
    ctx.set_precision("fp32c")
    got = run(ctx, full)
    assert close(got, ref)
with context(30) as ctx:
    run(ctx, ANY)
    before = used()
    want = ctx.td2(1)[0].copy()
    extra = used() - before
assert 0 < extra
with context(30) as ctx:
    run(ctx, ANY)
    shim.shim_limit(used() + extra - slots(2))
    assert np.array_equal(ctx.td2(1)[0], want)
print("done")
"""


def test_slots_take_only_what_is_left(tmp_path):
    src, lib = tmp_path / "shim.c", tmp_path / "libshim.so"
    src.write_text(SHIM)
    cudart = "libcudart.so." + torch.version.cuda.split(".")[0]
    subprocess.run(["gcc", "-O1", "-fPIC", "-shared", f'-DCUDART="{cudart}"', "-o", str(lib), str(src), "-ldl"], check=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    env = {**os.environ, "LD_PRELOAD": str(lib)}
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT, str(lib), str(sms)], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr
