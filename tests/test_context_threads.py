"""What contexts on several threads share: constant tables and kernel attributes.

gbfmm_create fills host tables and copies them to the device's constants; launches set kernels' limits
of dynamic shared memory.  Here the copies go to a stand-in that looks at the host table for a while,
as a slow copy would, and counts tables that change meanwhile or differ from the ones of the first
creation, and the limits to one that keeps what each kernel was given.  No GPU is seen: nothing is
launched.
"""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

COPY = r"""
#include <pthread.h>
#include <stdint.h>
#include <unistd.h>
static pthread_mutex_t mu = PTHREAD_MUTEX_INITIALIZER;
static struct { const void *sym; uint64_t hash; } seen[64];
static int nseen, bad, copies;
static uint64_t fnv(const unsigned char *p, size_t n)
{
    uint64_t h = 1469598103934665603ull;
    for (size_t i = 0; i < n; ++i) h = (h ^ ((const volatile unsigned char *)p)[i]) * 1099511628211ull;
    return h;
}
int __cudaLaunchKernel() { return 0; }
int cudaMemsetAsync() { return 0; }
int cudaMemcpyToSymbol(const void *sym, const void *src, size_t n, size_t offset, int kind)
{
    (void)offset, (void)kind;
    const uint64_t a = fnv(src, n);
    usleep(300);
    const uint64_t b = fnv(src, n);
    pthread_mutex_lock(&mu);
    int i = 0;
    while (i < nseen && seen[i].sym != sym) ++i;
    if (i == nseen) seen[nseen].sym = sym, seen[nseen++].hash = a;
    bad += a != b || a != seen[i].hash;
    ++copies;
    pthread_mutex_unlock(&mu);
    return 0;
}
static struct { const void *fn; int lo, hi; } limits[256];
static int nlimits;
int cudaFuncSetAttribute(const void *fn, int attr, int value)
{
    if (attr != 8) return 0; /* cudaFuncAttributeMaxDynamicSharedMemorySize */
    int i = 0;
    while (i < nlimits && limits[i].fn != fn) ++i;
    if (i == nlimits) limits[nlimits].fn = fn, limits[nlimits].lo = limits[nlimits].hi = value, ++nlimits;
    if (value < limits[i].lo) limits[i].lo = value;
    if (value > limits[i].hi) limits[i].hi = value;
    return 0;
}
int kernels_limited(void) { return nlimits; }
int kernels_changed(void)
{
    int c = 0;
    for (int i = 0; i < nlimits; ++i) c += limits[i].lo != limits[i].hi;
    return c;
}
int copies_made(void) { return copies; }
int copies_bad(void) { return bad; }
"""

RUN = r"""
import ctypes, sys, threading
copy, lib = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL), ctypes.CDLL(sys.argv[2])
init = [getattr(lib, f) for f in ("_ZN5gbfmm24init_expansion_constantsEv", "_ZN5gbfmm18init_m2l_constantsEv",
                                  "_ZN5gbfmm22init_m2l_f16_constantsEv", "_ZN5gbfmm22init_m2l_rot_constantsEv")]
def create():
    for f in init:
        f()
create()
first = copy.copies_made()
threads = [threading.Thread(target=lambda: [create() for _ in range(20)]) for _ in range(8)]
[t.start() for t in threads]
[t.join() for t in threads]
print(first, copy.copies_made(), copy.copies_bad())
"""


SORT = r"""
import ctypes, sys
copy, lib = ctypes.CDLL(sys.argv[1], mode=ctypes.RTLD_GLOBAL), ctypes.CDLL(sys.argv[2])
P = ctypes.c_void_p
for name in ("_ZN5gbfmm18launch_sort_gatherEPjS0_S0_S0_liPvPiPK6float4PS3_PS0_S7_P11CUstream_st",
             "_ZN5gbfmm20launch_sort_gather64EPmS0_PjS1_liPvPiPK6float4PS4_PS0_PS1_P11CUstream_st"):
    sort = getattr(lib, name)
    sort.restype, sort.argtypes = None, [P, P, P, P, ctypes.c_int64, ctypes.c_int] + 7 * [P]
    out = [ctypes.byref(ctypes.c_void_p()) for _ in range(2)]
    for n in (1000, 300_000, 1 << 20, 1 << 23):  # tiles of 1024, 2048, 4096 keys; passes that scan first
        sort(None, None, None, None, n, 30, None, None, None, None, *[ctypes.cast(o, P) for o in out], None)
print(copy.kernels_limited(), copy.kernels_changed())
"""


def run_with_stand_ins(tmp_path, script):
    from paper_1010_1482_gb300 import build

    lib = build.build()
    src, so = tmp_path / "copy.c", tmp_path / "copy.so"
    src.write_text(COPY)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(so), str(src), "-lpthread"], check=True)
    r = subprocess.run([sys.executable, "-c", script, str(so), lib], capture_output=True, text=True, cwd=ROOT,
                       env={**os.environ, "LD_PRELOAD": str(so), "CUDA_VISIBLE_DEVICES": ""}, timeout=300)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    return map(int, r.stdout.split())


def test_sorts_of_different_sizes_set_the_same_limits(tmp_path):
    """A sort that set another kernel's limit to its own tile's bytes made the launch of a larger sort on
    another thread fail."""
    limited, changed = run_with_stand_ins(tmp_path, SORT)
    assert limited == 8 and changed == 0, (limited, changed)


def test_tables_of_contexts_created_at_once(tmp_path):
    first, made, bad = run_with_stand_ins(tmp_path, RUN)
    assert first >= 8 and made == 161 * first and bad == 0, (first, made, bad)
