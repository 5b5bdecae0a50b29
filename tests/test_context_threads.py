"""Contexts created by several threads at once upload the same constant tables.

gbfmm_create fills host tables and copies them to the device's constants.  Here the copies go to a
stand-in that looks at the host table for a while, as a slow copy would, and counts tables that change
meanwhile or differ from the ones of the first creation.  No GPU is needed.
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


def test_tables_of_contexts_created_at_once(tmp_path):
    from paper_1010_1482_gb300 import build

    lib = build.build()
    src, so = tmp_path / "copy.c", tmp_path / "copy.so"
    src.write_text(COPY)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(so), str(src), "-lpthread"], check=True)
    r = subprocess.run([sys.executable, "-c", RUN, str(so), lib], capture_output=True, text=True, cwd=ROOT,
                       env={**os.environ, "LD_PRELOAD": str(so)}, timeout=300)
    if r.returncode != 0:
        pytest.fail(r.stderr)
    first, made, bad = map(int, r.stdout.split())
    assert first >= 8 and made == 161 * first and bad == 0, (first, made, bad)
