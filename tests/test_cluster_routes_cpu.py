"""Which kernels a call launches, also on a GPU that holds fewer thread-block
clusters, or none, or cannot say: the CUDA runtime is replaced by a fake that
records launches (nothing runs), so no GPU is needed."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <string.h>
typedef struct { unsigned x, y, z; } dim3_;
typedef struct { int id; char pad[4]; union { char b[64]; dim3_ d; } val; } attr_;
typedef struct { dim3_ grid, block; size_t smem; void *stream; attr_ *attrs; unsigned n; } cfg_;
static int device, last, clusters[64], log_[256], count;
void fake_reset(int dev) { device = dev; count = 0; }
void fake_clusters(int dev, int n) { clusters[dev] = n; }  /* -1: the query fails */
int fake_last(void) { return last; }
int fake_log(int *out) { memcpy(out, log_, sizeof(int) * count); return count; }
static int fail(int e) { return last = e; }
int cudaGetDevice(int *d) { *d = device; return 0; }
int cudaDeviceGetAttribute(int *v, int a, int d) { *v = 152; return 0; }
int cudaFuncSetAttribute(const void *f, int a, int v) { return 0; }
int cudaGetLastError(void) { int e = last; last = 0; return e; }
int cudaMemsetAsync(void *p, int v, size_t n, void *s) { return 0; }
int cudaOccupancyMaxActiveClusters(int *n, const void *f, const cfg_ *c) {
  if (clusters[device] < 0) return fail(1);
  *n = clusters[device];
  if (*n == 999) {  /* a whole chip's counts */
    const int size = (int)c->attrs[0].val.d.x;
    *n = size == 2 ? 76 : size == 4 ? 36 : size == 8 ? 15 : 1;
  }
  return 0;
}
int cudaLaunchKernelExC(const cfg_ *c, const void *f, void **args) {
  int size = 1;
  for (unsigned i = 0; i < c->n; ++i)
    if (c->attrs[i].id == 4) size = (int)c->attrs[i].val.d.x;  /* cudaLaunchAttributeClusterDimension */
  if (size > 1 && clusters[device] < 1) return fail(701);
  log_[count++] = size;
  return 0;
}
int __cudaPushCallConfiguration(dim3_ g, dim3_ b, size_t m, void *s) { return 0; }
int __cudaPopCallConfiguration(dim3_ *g, dim3_ *b, size_t *m, void *s) { return 0; }
int __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
int __cudaLaunchKernel(void *k, dim3_ g, dim3_ b, void **args, size_t m, void *s) { log_[count++] = 1; return 0; }
static int encode(void *map) { memset(map, 0, 128); return 0; }
int cudaGetDriverEntryPointByVersion(const char *n, void **fn, unsigned v, unsigned long long f, int *q) {
  *fn = (void *)encode; *q = 0;
  return 0;
}
"""

RUN = r"""
import ctypes, json, sys
sys.path.insert(0, sys.argv[1])
from paper_2609_09240_gb300 import tq
L, F = tq.lib(), ctypes.CDLL(None)
p = lambda i: ctypes.c_void_p(0x10000 * (i + 1))  # never dereferenced

def ternarize(N, K, nnz):
    return L.tq_ternarize(N, K, p(0), nnz, 4, p(1), p(2), p(3), p(4), p(5), p(6), p(7), p(8), 1 << 40, p(9), None)

def prefill(M, N, K, nnz=0):
    w = tq.tq_weight()
    w.N, w.K, w.group, w.nnz = N, K, 128, nnz
    w.plane1 = w.salience = w.rowptr = w.scale1 = w.offset = w.plane2 = w.scale2 = w.p2index = 0x10000
    return L.tq_linear(M, N, K, ctypes.byref(w), p(0), p(1), p(2), 1 << 40, None)

out = []
for dev, clusters, call in json.loads(sys.argv[2]):
    F.fake_clusters(dev, clusters)
    F.fake_reset(dev)
    rc = {"ternarize": ternarize, "prefill": prefill, "linear": prefill}[call[0]](*call[1:])
    log = (ctypes.c_int * 256)()
    n = F.fake_log(log)
    out.append([rc, list(log[:n]), F.fake_last()])
print("OUT" + json.dumps(out))
"""


@pytest.fixture(scope="module")
def launches(tmp_path_factory):
    from paper_2609_09240_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("fake")
    (d / "fake.c").write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(d / "fake.so"), str(d / "fake.c")], check=True)

    def run(*steps):
        r = subprocess.run([sys.executable, "-c", RUN, ROOT, json.dumps(steps)], capture_output=True, text=True,
                           env=dict(os.environ, LD_PRELOAD=str(d / "fake.so")))
        assert r.returncode == 0, r.stderr
        return json.loads(r.stdout.split("OUT")[1])
    return run


def test_prefill_splits_only_where_clusters_run(launches):
    call = ("prefill", 64, 1024, 4096)  # eight tiles
    (one, no, failed, other) = launches((0, 15, call), (1, 0, call), (2, -1, call), (3, 36, call))
    assert one == [0, [8], 0] and other == [0, [8], 0]
    assert no == [0, [1], 0]
    assert failed == [0, [1], 0]  # the query's error is not the call's
    assert launches((0, -1, call)) == [[0, [1], 0]]


def test_prefill_splits_only_where_it_saves_groups(launches):
    shapes = [((256, 640, 512), 1), ((256, 640, 896), 1),   # two and three groups saved
              ((128, 1024, 1024), 4), ((128, 1024, 2048), 8),
              ((512, 4096, 1280), 1), ((512, 4096, 1536), 1), ((512, 4096, 1792), 2),  # 64 tiles
              ((200, 9728, 2560), 2), ((200, 19456, 2560), 1)]
    got = launches(*[(0, 999, ("prefill", *shape)) for shape, _ in shapes])
    assert got == [[0, [split], 0] for _, split in shapes]


def test_ternarize_selects_without_a_cluster(launches):
    """Statistics, selection, planes: one cluster of 16 where the device holds
    one, else the whole chip's kernels (four digits, count, mark, rowptr)."""
    call = ("ternarize", 256, 1024, 200)
    (one, no, failed, other) = launches((0, 1, call), (1, 0, call), (2, -1, call), (3, 1, call))
    assert one == [0, [1, 16, 1], 0] and other == [0, [1, 16, 1], 0]
    assert no == [0, [1] * 9, 0] and failed == [0, [1] * 9, 0]
    too_many = ("ternarize", 26609, 128, 200)  # keys beyond the cluster's shared memory
    assert launches((0, 1, too_many)) == [[0, [1] * 9, 0]]


def test_one_token_planes_in_one_kernel(launches):
    """Prep and one kernel for both planes, or prep, second plane, first plane:
    few salient groups in many stages take the two kernels."""
    salient = lambda N, K, share: int(N * (K // 128) * share)
    cases = [((1, 2560, 4096, 1), 2), ((1, 4096, 12288, salient(4096, 12288, 1.0)), 2),
             ((1, 49152, 4096, salient(49152, 4096, 0.1)), 2), ((1, 49152, 4096, salient(49152, 4096, 0.01)), 3),
             ((1, 151936, 4096, salient(151936, 4096, 0.3)), 2), ((1, 151936, 4096, salient(151936, 4096, 0.01)), 3),
             ((1, 40000, 8192, 15000 * 11), 2), ((1, 40000, 8192, 15000 * 11 - 1), 3),  # 16 stages on the busiest SM
             ((1, 200000, 4096, salient(200000, 4096, 0.3)), 3),  # more than 16 on every SM
             ((1, 2560, 4096, 0), 2)]  # no second plane
    got = launches(*[(0, 0, ("linear", *args)) for args, _ in cases])
    assert got == [[0, [1] * n, 0] for _, n in cases]
