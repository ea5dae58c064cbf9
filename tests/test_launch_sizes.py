"""Host side of the network features' launches on devices and partitions smaller than the whole GPU, on the CPU:
the library runs against a fake CUDA runtime that answers size queries as told and records launches."""
import os
import subprocess
import sys

import pytest

import paper_1908_00210_gb300 as P

FAKE = r"""
#include <stddef.h>
#include <stdio.h>
#include <stdlib.h>
typedef struct { unsigned x, y, z; } d3;
static d3 grid0, block0; static size_t smem0; static void *stream0;
static int num(const char *n) { return atoi(getenv(n)); }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { *v = a == 16 ? num("SMS") : 0; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessor(int *n, const void *f, int b, size_t s) { *n = num("PER_SM"); return 0; }
int cudaOccupancyMaxActiveClusters(int *n, const void *f, const void *c) { *n = num("CLUSTERS"); return 0; }
int cudaGetLastError(void) { return 0; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
unsigned __cudaPushCallConfiguration(d3 g, d3 b, size_t s, void *st) { grid0 = g; block0 = b; smem0 = s; stream0 = st; return 0; }
int __cudaPopCallConfiguration(d3 *g, d3 *b, size_t *s, void *st) { *g = grid0; *b = block0; *s = smem0; *(void **)st = stream0; return 0; }
static int plain(d3 g, d3 b) {
    if (b.x == 1024 && g.x % 8 == 0 && num("CLUSTERS") < 1) return 912;              /* cudaErrorInvalidClusterSize */
    printf("%s %u\n", b.x == 1024 && g.x % 8 == 0 ? "cluster" : "plain", g.x);
    return 0;
}
int __cudaLaunchKernel(void *k, d3 g, d3 b, void **a, size_t s, void *st) { return plain(g, b); }
int cudaLaunchKernel(const void *k, d3 g, d3 b, void **a, size_t s, void *st) { return plain(g, b); }
int cudaLaunchKernelExC(const d3 *cfg, const void *f, void **a) { return plain(cfg[0], cfg[1]); }
int cudaLaunchCooperativeKernel(const void *f, d3 g, d3 b, void **a, size_t s, void *st) {
    if ((int)g.x > num("SMS") * num("PER_SM")) return 720;                           /* cudaErrorCooperativeLaunchTooLarge */
    printf("cooperative %u\n", g.x);
    return 0;
}
"""
CALL = """
import ctypes as C, sys
f = C.CDLL(sys.argv[1]).gdi_mpnn_features
f.argtypes = [C.c_int64, C.c_int32] + [C.c_void_p] * 4 + [C.c_uint64, C.c_int32, C.c_int32] + [C.c_void_p] * 3
p = 4096                       # never read: nothing runs
print('rc', f(2000, 1, p, p, p, p, 7, int(sys.argv[2]), 0, p, p, None))
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    subprocess.check_call(["gcc", "-shared", "-fPIC", "-o", str(d / "fake.so"), str(d / "fake.c")])
    lib = P.build()

    def call(steps, **env):
        out = subprocess.check_output([sys.executable, "-c", CALL, lib, str(steps)], text=True,
                                      env=dict(os.environ, LD_PRELOAD=str(d / "fake.so"), **{k: str(v) for k, v in env.items()}))
        lines = out.split("\n")[:-1]
        assert "rc 0" in lines, lines
        return [x for x in lines if not x.startswith("rc")]
    return call


@pytest.mark.parametrize("sms,per_sm", [(152, 4), (152, 2), (148, 4), (76, 4), (16, 3), (1, 1)])
def test_walk_fits_the_device(fake, sms, per_sm):
    """One cluster launch, and a cooperative one of no more blocks than the device holds."""
    got = dict(x.split() for x in fake(256, SMS=sms, PER_SM=per_sm, CLUSTERS=2))
    assert got["cluster"] == "8" and 1 <= int(got["cooperative"]) <= sms * per_sm


def test_walk_without_clusters(fake):
    """A partition that holds no cluster of eight walks with one launch per step."""
    got = fake(256, SMS=4, PER_SM=4, CLUSTERS=0)
    assert len(got) == 1 + 256 + 1 and all(x.startswith("plain") for x in got)
