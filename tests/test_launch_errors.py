"""Launch errors of the proposal network's calls, without a GPU: a small
stand-in for the CUDA runtime (preloaded in a child process) keeps "device"
memory on the host, runs no kernel and refuses the launch it is told to.
Every call must report the refused launch, whichever it is, and leave no error
behind for the next call; an output at an address that no kernel can store a
float to is written by a copy; the grids follow the device's number of
multiprocessors."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <stdlib.h>
#include <string.h>
typedef int err;                     /* cudaError_t: 0 success, 719 launch failure */
typedef struct { unsigned x, y, z; } dim3_;
static int refuse = -1, seen = 0, last = 0;
static const void *odd = 0;          /* an address only copies may write */
static int copied = 0;
void fake_watch(const void *p) { odd = p; copied = 0; }
int fake_copied(void) { return copied; }
void fake_refuse(int k) { refuse = k; seen = 0; }
int fake_launches(void) { return seen; }
/* the error of the launch, which the runtime keeps until it is asked for */
static int sms = 152, grids[64];
void fake_sms(int n) { sms = n; }
int fake_grid(int k) { return grids[k]; }
static err launch(unsigned grid)
{
    if (seen < 64) grids[seen] = (int)grid;
    if (seen++ == refuse) { last = 719; return 719; }
    return 0;
}
err cudaMalloc(void **p, size_t n) { *p = calloc(n, 1); return 0; }
err cudaFree(void *p) { free(p); return 0; }
err cudaMemset(void *p, int v, size_t n) { memset(p, v, n); return 0; }
err cudaMemcpy(void *d, const void *s, size_t n, int k) { (void)k; memcpy(d, s, n); return 0; }
err cudaMemcpyAsync(void *d, const void *s, size_t n, int k, void *st)
{ (void)k; (void)st; if (d == odd) copied = 1; memcpy(d, s, n); return 0; }
err cudaGetDevice(int *d) { *d = 0; return 0; }
err cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = sms; return 0; }
err cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
err cudaDeviceSynchronize(void) { return 0; }
err cudaStreamSynchronize(void *s) { (void)s; return 0; }
err cudaGetLastError(void) { err e = last; last = 0; return e; }
const char *cudaGetErrorString(err e) { return e ? "launch failure" : "no error"; }
err __cudaGetKernel(void **k, const void *f) { *k = (void *)f; return 0; }
err __cudaLaunchKernel(void *k, dim3_ g, dim3_ b, void **a, size_t m, void *s)
{ (void)k; (void)b; (void)a; (void)m; (void)s; return launch(g.x); }
err cudaLaunchKernel(const void *f, dim3_ g, dim3_ b, void **a, size_t m, void *s)
{ (void)f; (void)b; (void)a; (void)m; (void)s; return launch(g.x); }
err cudaLaunchKernelExC(const void *c, const void *f, void **a) { (void)f; (void)a; return launch(*(const unsigned *)c); }   /* gridDim comes first */
"""

CHILD = r"""
import ctypes
import sys

import numpy as np

sys.path.insert(0, ".")
import paper_2607_16897_gb300 as glt

fake = ctypes.CDLL(sys.argv[1])
fake.fake_watch.argtypes = [ctypes.c_void_p]
B, mode = int(sys.argv[2]), sys.argv[3]
if mode == "grids":
    fake.fake_sms(37)
net = glt.NN(B, np.zeros(glt.GLT_NN_PARAMS, np.float32))
x, m, t, y = (np.zeros((B, k), np.float32) for k in (1200, 6, 8, 8))
p = [a.ctypes.data for a in (x, m, t, y)]
loss = np.zeros(2, np.float32)
calls = {"forward": lambda: net.forward(p[0], p[1], p[3], B, stream=0),
         "gradient": lambda: net.gradient(p[0], p[1], p[2], B, stream=0),
         "train_step": lambda: net.train_step(p[0], p[1], p[2], B, 1e-3, loss.ctypes.data, stream=0)}
for name, call in calls.items() if mode == "launches" else ():
    fake.fake_refuse(-1)
    call()
    n = fake.fake_launches()
    assert n >= 2, (name, n)
    for k in range(n):
        fake.fake_refuse(k)
        try:
            call()
            print("no error from", name, "launch", k, "of", n)
        except glt.GltError as e:
            assert "launch failure" in str(e), e
        fake.fake_refuse(-1)
        try:
            call()
        except glt.GltError as e:
            print("error left behind by", name, "launch", k, "of", n)
            fake.cudaGetLastError()
raw = np.zeros(B * 8 * 4 + 8, np.uint8)
for off in (0, 1, 2, 3) if mode == "addresses" else ():
    a = (raw.ctypes.data + 3) // 4 * 4 + off
    for name, call in (("forward", lambda: net.forward(p[0], p[1], a, B, stream=0)),
                       ("train_step", lambda: net.train_step(p[0], p[1], p[2], B, 1e-3, a, stream=0))):
        fake.fake_watch(a)
        call()
        if off and not fake.fake_copied():
            print("a kernel stores the output of", name, "at offset", off)
if mode == "grids":
    fake.fake_refuse(-1)
    calls["train_step"]()
    g = [fake.fake_grid(k) for k in range(fake.fake_launches())]
    if g.count(min(B, 37)) != 3:          # forward, input gradient, weight gradient of the convolutions
        print("grids of a training step of", B, "samples on 37 multiprocessors:", g)
print("done")
"""


def run_child(tmp_path, B, mode):
    import importlib.util
    spec = importlib.util.spec_from_file_location("_glt_build", os.path.join(ROOT, "paper_2607_16897_gb300", "build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.build()
    src, lib = tmp_path / "fake.c", str(tmp_path / "fake.so")
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", lib, str(src)], check=True)
    env = dict(os.environ, LD_PRELOAD=lib)
    env.pop("GLT_LIBRARY", None)
    r = subprocess.run([sys.executable, "-c", CHILD, lib, str(B), mode], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.split("\n")[:-1] == ["done"], r.stdout + r.stderr[-2000:]


@pytest.mark.parametrize("B", [5, 2100])
def test_refused_launches_are_reported(tmp_path, B):
    run_child(tmp_path, B, "launches")


@pytest.mark.parametrize("B", [5, 2100])
def test_outputs_at_any_address(tmp_path, B):
    run_child(tmp_path, B, "addresses")


@pytest.mark.parametrize("B", [150, 2100])
def test_convolutions_take_a_block_per_multiprocessor(tmp_path, B):
    run_child(tmp_path, B, "grids")
