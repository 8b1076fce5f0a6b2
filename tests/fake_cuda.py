"""A second copy of the library whose copies and time-out reads the tests can make fail.

The library's objects are linked once more with cudaMemcpy and
cudaMemcpyFromSymbolAsync wrapped (ld --wrap): the copy with index
``fail_copy`` since the last reset is not made and returns an error, and with
``timed_out`` set the time-out flag reads as set.  Everything fails on the
host: nothing reaches the GPU that an undisturbed call would not send."""
import contextlib
import ctypes as C
import glob
import os
import subprocess

from paper_2405_04229_gb300 import binding as B
from paper_2405_04229_gb300 import build

_SHIM = r"""
int fake_fail_copy = -1, fake_copies = 0, fake_timed_out = 0;
int __real_cudaMemcpy(void*, const void*, unsigned long, int);
int __wrap_cudaMemcpy(void* d, const void* s, unsigned long n, int kind) {
    if (fake_copies++ == fake_fail_copy) return 999; /* cudaErrorUnknown */
    return __real_cudaMemcpy(d, s, n, kind);
}
int __real_cudaMemcpyFromSymbolAsync(void*, const void*, unsigned long, unsigned long, int, void*);
int __wrap_cudaMemcpyFromSymbolAsync(void* d, const void* s, unsigned long n, unsigned long off, int kind, void* stream) {
    const int e = __real_cudaMemcpyFromSymbolAsync(d, s, n, off, kind, stream);
    if (fake_timed_out) *(unsigned int*)d = 1u; /* (a copy to pageable memory is complete on return) */
    return e;
}
"""


def link(folder):
    """Links the library with the wrapped calls into `folder`; returns its path."""
    build.build()
    src, obj, lib = (os.path.join(folder, f) for f in ("shim.c", "shim.o", "libcherenkov_fake.so"))
    with open(src, "w") as f:
        f.write(_SHIM)
    subprocess.run(["gcc", "-O1", "-fPIC", "-c", src, "-o", obj], check=True)
    objs = [os.path.join(build.OBJ_DIR, os.path.basename(s)[:-3] + ".o") for s in build._sources()]
    assert all(o in glob.glob(os.path.join(build.OBJ_DIR, "*.o")) for o in objs)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", lib, *objs, obj, "-Xlinker", "--wrap=cudaMemcpy",
                    "-Xlinker", "--wrap=cudaMemcpyFromSymbolAsync", "-lcudart_static", "-lrt", "-lpthread", "-ldl"],
                   check=True)
    return lib


class Fake:
    def __init__(self, L):
        self._v = {k: C.c_int.in_dll(L, "fake_" + k) for k in ("fail_copy", "copies", "timed_out")}

    def reset(self, fail_copy=-1, timed_out=0):
        self._v["fail_copy"].value, self._v["copies"].value, self._v["timed_out"].value = fail_copy, 0, timed_out

    @property
    def copies(self):
        return self._v["copies"].value


@contextlib.contextmanager
def loaded(path):
    """The binding on the wrapped library for the duration of the block; yields its Fake."""
    lib, where = B._lib, B._LIB_PATH
    B._lib, B._LIB_PATH = None, path
    try:
        fake = Fake(B.lib())
        yield fake
        fake.reset()
    finally:
        B._lib, B._LIB_PATH = lib, where
