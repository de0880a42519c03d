"""A grid that releases its dependents at once and stores only some time later, as a caller's own
kernel with programmatic dependent launch may: what it writes is there for the library's kernels
only if they wait for the whole grid.  Compiled with nvcc on first use."""
import ctypes
import os
import subprocess
import tempfile

from paper_2607_02963_gb300 import build

SOURCE = r"""
#include <cuda_runtime.h>
#include <stdint.h>
struct Copies { uint4* dst[8]; const uint4* src[8]; unsigned long long n16[8]; int n; };
__device__ unsigned long long now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__global__ void late_store(const __grid_constant__ Copies c, unsigned delay_ns) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned long long t0 = now();
  for (int i = 0; i < 1000000 && now() - t0 < delay_ns; ++i) __nanosleep(200);  // (bounded)
  for (int k = 0; k < c.n; ++k)
    for (unsigned long long i = blockIdx.x * blockDim.x + threadIdx.x; i < c.n16[k]; i += gridDim.x * blockDim.x)
      c.dst[k][i] = c.src[k][i];
}
extern "C" int late_store_launch(void** dst, void** src, unsigned long long* bytes, int n, unsigned delay_ns, void* stream) {
  Copies c = {};
  if (n < 0 || n > 8) return 1;
  for (c.n = 0; c.n < n; ++c.n) {
    if (bytes[c.n] % 16 || (uintptr_t)dst[c.n] % 16 || (uintptr_t)src[c.n] % 16) return 1;
    c.dst[c.n] = (uint4*)dst[c.n];
    c.src[c.n] = (const uint4*)src[c.n];
    c.n16[c.n] = bytes[c.n] / 16;
  }
  late_store<<<8, 256, 0, (cudaStream_t)stream>>>(c, delay_ns);
  return (int)cudaGetLastError();
}
"""

_lib = None


def _load():
    global _lib
    if _lib is None:
        tmp = tempfile.mkdtemp(prefix="late_writer_")
        cu, so = os.path.join(tmp, "late_writer.cu"), os.path.join(tmp, "late_writer.so")
        with open(cu, "w") as f:
            f.write(SOURCE)
        subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-shared", "-Xcompiler", "-fPIC", cu, "-o", so], check=True)
        _lib = ctypes.CDLL(so)
    return _lib


def late_store(pairs, stream, delay_us=100):
    """Enqueue dst <- src for (dst, src) pairs of equally sized device tensors, stored ``delay_us`` after
    the grid has released its dependents."""
    n = len(pairs)
    ptrs = [(ctypes.c_void_p * n)(*[p[i].data_ptr() for p in pairs]) for i in (0, 1)]
    size = [d.numel() * d.element_size() for d, _ in pairs]
    assert size == [s.numel() * s.element_size() for _, s in pairs]
    st = _load().late_store_launch(ptrs[0], ptrs[1], (ctypes.c_ulonglong * n)(*size), n, int(1000 * delay_us),
                                   ctypes.c_void_p(stream.cuda_stream))
    assert st == 0, f"late_store_launch: {st}"
