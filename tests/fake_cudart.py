"""The library's objects linked against a CUDA runtime that only keeps count, so
that its host code runs without a GPU: kernels are not run, memory is malloc'ed,
and a test says what a call of the runtime returns.  A device variable's value is
that of its host shadow."""
import ctypes
import os
import subprocess

from paper_2105_07298_gb300 import build as apsp_build

# Calls that do more than return `error` (0 unless a test sets it).
_SRC = r"""
#include <stdlib.h>
#include <string.h>
int capturing, pool_error, pool_attr_error, alloc_error;
int programmatic, launches, copies, memsets, pools_created, pools_destroyed, pools_trimmed, pool_allocs, allocs, frees, live;
static void *vars[256]; static const char *names[256]; int num_vars;
void *var_at(int i) { return vars[i]; }
const char *var_name(int i) { return names[i]; }
int cudaGetDevice(int *d) { *d = 0; return 0; }
int cudaDeviceGetAttribute(int *v, int attr, int dev) { *v = 152; return 0; }
int cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *v) { *v = 3; return 0; }
int cudaStreamIsCapturing(void *s, int *st) { *st = capturing ? 1 : 0; return 0; }
static int take(void **p, size_t n) { *p = malloc(n); ++live; return 0; }
int cudaMalloc(void **p, size_t n) { return take(p, n); }
int cudaMallocAsync(void **p, size_t n, void *s) { ++allocs; return alloc_error ? alloc_error : take(p, n); }
int cudaMallocFromPoolAsync(void **p, size_t n, void *pool, void *s) {
  ++pool_allocs;
  return pool_error ? pool_error : take(p, n);
}
int cudaFree(void *p) { if (p) --live; free(p); return 0; }
int cudaFreeAsync(void *p, void *s) { ++frees; --live; free(p); return 0; }
int cudaMemPoolCreate(void **pool, const void *props) { *pool = malloc(1); ++pools_created; return 0; }
int cudaMemPoolDestroy(void *pool) { ++pools_destroyed; free(pool); return 0; }
int cudaMemPoolTrimTo(void *pool, size_t keep) { ++pools_trimmed; return 0; }
int cudaMemPoolSetAttribute(void *pool, int attr, void *v) { return pool_attr_error; }
int cudaMemcpyAsync(void) { ++copies; return 0; }
int cudaMemsetAsync(void) { ++memsets; return 0; }
int cudaMemcpyFromSymbol(void *d, const char *s, size_t n, size_t at) { memcpy(d, s + at, n); return 0; }
int cudaMemcpyToSymbol(char *s, const void *d, size_t n, size_t at) { memcpy(s + at, d, n); return 0; }
int cudaGetSymbolAddress(void **p, void *s) { *p = s; return 0; }
int cudaStreamCreateWithPriority(void **s) { *s = (void *)1; return 0; }
int cudaEventCreateWithFlags(void **e) { *e = (void *)1; return 0; }
int cudaEventCreate(void **e) { *e = (void *)1; return 0; }
int cudaEventElapsedTime(float *ms) { *ms = 1.0f; return 0; }
int __cudaLaunchKernel(void) { ++launches; return 0; }
struct config { unsigned grid[3], block[3]; size_t smem; void *stream; int *attrs; unsigned num; };
int cudaLaunchKernelExC(const struct config *c) { /* attribute 6: may start before its predecessor ends */
  for (unsigned i = 0; i < c->num; ++i) programmatic += c->attrs[18 * i] == 6;
  ++launches;
  return 0;
}
static int fatbin;
void **__cudaRegisterFatBinary(void *f) { return (void **)&fatbin; }
void __cudaRegisterVar(void **f, void *host, char *dev, const char *name) {
  vars[num_vars] = host;
  names[num_vars++] = name;
}
"""


def load(tmp_path):
    """A fresh copy of the library on the counting runtime."""
    apsp_build.build()
    objs = [os.path.join(apsp_build.OUT_DIR, f) for f in sorted(os.listdir(apsp_build.OUT_DIR)) if f.endswith(".o")]
    srcs = {f[:-3] for f in os.listdir(apsp_build.CSRC) if f.endswith(".cu")}
    objs = [o for o in objs if os.path.basename(o)[:-2] in srcs]
    nm = subprocess.run(["nm", "-u", *objs], capture_output=True, text=True, check=True).stdout
    wanted = {w for w in nm.split() if w.startswith(("cuda", "__cuda"))}
    rest = [w for w in sorted(wanted) if f" {w}(" not in _SRC.replace("*", " ")]
    src = tmp_path / "cudart.c"
    src.write_text(_SRC + "".join(f"long {w}(void) {{ return 0; }}\n" for w in rest))
    so = tmp_path / "libapspfw_host.so"
    subprocess.run(["gcc", "-w", "-O1", "-fPIC", "-c", str(src), "-o", str(tmp_path / "cudart.o")], check=True)
    subprocess.run(["gcc", "-shared", "-Wl,-Bsymbolic", "-o", str(so), *objs, str(tmp_path / "cudart.o"), "-lstdc++"],
                   check=True)
    lib = ctypes.CDLL(str(so))
    lib.var_at.restype = ctypes.c_void_p
    lib.var_name.restype = ctypes.c_char_p
    return lib


def word(lib, name):
    """One of the runtime's counters or switches."""
    return ctypes.c_int.in_dll(lib, name)
