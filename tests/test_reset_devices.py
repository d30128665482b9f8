"""Resets on a device or stream that is not the tables': the library runs
against a fake of the CUDA runtime calls that a reset makes (two devices, host
memory), so that no GPU is needed."""
import os
import subprocess
import sys

import pytest

from paper_2607_03441_gb300 import build

# A stream is (device + 1) << 32; the null stream belongs to the current device.
FAKE = r"""
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
static int cur, memsets, launches;
void fake_set(int dev) { cur = dev; memsets = launches = 0; }
int fake_memsets(void) { return memsets; }
int fake_launches(void) { return launches; }
static int dev_of(void *s) { return s ? (int)((uintptr_t)s >> 32) - 1 : cur; }
int cudaGetDevice(int *d) { *d = cur; return 0; }
static int stream_ctx(void *s, void **c) { *c = (void *)(uintptr_t)(dev_of(s) + 1); return 0; }
static int current_ctx(void **c) { *c = (void *)(uintptr_t)(cur + 1); return 0; }
int cudaGetDriverEntryPointByVersion(const char *name, void **f, unsigned v, unsigned long long flags, int *q) {
    *f = !strcmp(name, "cuStreamGetCtx") ? (void *)stream_ctx : !strcmp(name, "cuCtxGetCurrent") ? (void *)current_ctx : 0;
    *q = *f ? 0 : 1;
    return 0;
}
int cudaDeviceGetAttribute(int *v, int attr, int dev) { *v = attr == 75 ? 10 : attr == 76 ? 3 : 152; return 0; }
int cudaMalloc(void **p, size_t n) { *p = aligned_alloc(256, (n + 255) / 256 * 256); return 0; }
int cudaFree(void *p) { free(p); return 0; }
int cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return 0; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { memset(p, v, n); ++memsets; return 0; }
int cudaDeviceSynchronize(void) { return 0; }
int cudaGetLastError(void) { return 0; }
/* a kernel launch: from a stream of another device it is refused (400) */
int cudaLaunchKernelExC(const void *cfg, const void *f, void **args) {
    void *stream;
    memcpy(&stream, (const char *)cfg + 32, sizeof stream); /* after two dim3 and the shared memory's size */
    if (dev_of(stream) != cur) return 400;
    ++launches;
    return 0;
}
"""

PROBE = r"""
import ctypes, sys
fake, lib = ctypes.CDLL(sys.argv[1]), ctypes.CDLL(sys.argv[2])
P = ctypes.c_void_p
stream_of = lambda dev: (dev + 1) << 32
fake.fake_set(0)
h, s = P(), P()
assert lib.attt_history_create(3, ctypes.c_int64(1000), ctypes.byref(h)) == 0
assert lib.attt_wordsets_create(70, ctypes.c_int64(5000), ctypes.byref(s)) == 0
for cur, stream in ((0, stream_of(0)), (0, 0), (1, stream_of(0)), (0, stream_of(1)), (1, stream_of(1)), (1, 0)):
    for name, reset, handle in (("history", lib.attt_history_reset, h), ("wordsets", lib.attt_wordsets_reset, s)):
        fake.fake_set(cur)
        print(name, reset(handle, P(stream)), fake.fake_launches(), fake.fake_memsets())
"""


@pytest.fixture(scope="module")
def resets(tmp_path_factory):
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(d / "fake.so"), str(d / "fake.c")], check=True)
    env = dict(os.environ, LD_PRELOAD=str(d / "fake.so"))
    out = subprocess.run([sys.executable, "-c", PROBE, str(d / "fake.so"), build.build()], env=env, check=True,
                         capture_output=True, text=True).stdout
    return [(w[0], *(int(v) for v in w[1:])) for w in (line.split() for line in out.splitlines())]


def test_resets_run_from_any_device_and_stream(resets):
    """(status, kernel launches, memsets) of each reset: a kernel where the
    tables, the current device and the stream's are one, memsets elsewhere."""
    assert len(resets) == 12
    here, elsewhere = resets[:4], resets[4:]
    assert here == [("history", 0, 1, 0), ("wordsets", 0, 1, 0)] * 2
    assert elsewhere == [("history", 0, 0, 1), ("wordsets", 0, 0, 2)] * 4
