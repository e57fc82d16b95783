"""A stand-in for single calls of the CUDA runtime, for tests of what the
library does when one of them fails: a small shared object, put before the
runtime (LD_PRELOAD) in a process of its own, that passes every call on unless
the test has armed a failure or a count.  Nothing fails on the GPU."""
import os
import subprocess
import sys
import textwrap

SOURCE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static void* real(const char* name) {
    void* lib = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    return lib ? dlsym(lib, name) : NULL;
}
/* cudaMalloc: out of memory for sizes from fake_malloc_max on (0: never), after
   fake_malloc_after more calls of at least fake_malloc_min bytes */
size_t fake_malloc_max = 0, fake_malloc_min = 0;
long fake_malloc_after = -1, fake_mallocs_refused = 0;
int cudaMalloc(void** p, size_t n) {
    static int (*f)(void**, size_t);
    if (!f) f = (int (*)(void**, size_t))real("cudaMalloc");
    int no = fake_malloc_max && n >= fake_malloc_max;
    if (fake_malloc_after >= 0 && n >= fake_malloc_min) {
        if (fake_malloc_after == 0) no = 1;
        else --fake_malloc_after;
    }
    if (no) { ++fake_mallocs_refused; return 2; }
    return f(p, n);
}
/* fake_capture: 1 cudaStreamBeginCapture fails, 2 cudaStreamEndCapture reports
   an invalidated capture (which has ended), 3 cudaGraphInstantiate fails */
int fake_capture = 0, fake_captures_refused = 0;
int cudaStreamBeginCapture(void* st, int mode) {
    static int (*f)(void*, int);
    if (!f) f = (int (*)(void*, int))real("cudaStreamBeginCapture");
    if (fake_capture == 1) { ++fake_captures_refused; return 900; }
    return f(st, mode);
}
int cudaStreamEndCapture(void* st, void** g) {
    static int (*f)(void*, void**);
    if (!f) f = (int (*)(void*, void**))real("cudaStreamEndCapture");
    const int e = f(st, g);
    if (fake_capture == 2) { ++fake_captures_refused; *g = NULL; return 901; }
    return e;
}
int cudaGraphInstantiate(void** x, void* g, unsigned long long flags) {
    static int (*f)(void**, void*, unsigned long long);
    if (!f) f = (int (*)(void**, void*, unsigned long long))real("cudaGraphInstantiate");
    if (fake_capture == 3) { ++fake_captures_refused; return 2; }
    return f(x, g, flags);
}
/* fake_device >= 0: the number that cudaGetDevice gives for the one device there
   is; func_attributes: calls of cudaFuncSetAttribute */
int fake_device = -1;
long func_attributes = 0;
int cudaGetDevice(int* d) {
    static int (*f)(int*);
    if (!f) f = (int (*)(int*))real("cudaGetDevice");
    const int e = f(d);
    if (fake_device >= 0) *d = fake_device;
    return e;
}
int cudaDeviceGetAttribute(int* v, int attr, int dev) {
    static int (*f)(int*, int, int);
    if (!f) f = (int (*)(int*, int, int))real("cudaDeviceGetAttribute");
    return f(v, attr, fake_device >= 0 && dev == fake_device ? 0 : dev);
}
/* fake_clusters >= 0: the clusters that run at once */
int fake_clusters = -1;
int cudaOccupancyMaxActiveClusters(int* n, const void* fn, const void* cfg) {
    static int (*f)(int*, const void*, const void*);
    if (!f) f = (int (*)(int*, const void*, const void*))real("cudaOccupancyMaxActiveClusters");
    const int e = f(n, fn, cfg);
    if (fake_clusters >= 0) *n = fake_clusters;
    return e;
}
int cudaFuncSetAttribute(const void* fn, int attr, int v) {
    static int (*f)(const void*, int, int);
    if (!f) f = (int (*)(const void*, int, int))real("cudaFuncSetAttribute");
    ++func_attributes;
    return f(fn, attr, v);
}
"""


def run(tmp_path, code, timeout=300):
    """Run `code` (with `lib`, the ctypes handle of the stand-in) in a fresh
    python of this repository; returns its output, raises when it fails."""
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    here = os.path.dirname(os.path.abspath(__file__))
    head = "import ctypes, sys\nsys.path[:0] = [%r, %r]\nlib = ctypes.CDLL(%r)\n" % (os.path.dirname(here), here, str(so))
    r = subprocess.run([sys.executable, "-c", head + textwrap.dedent(code)], capture_output=True, text=True,
                       timeout=timeout, env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout
