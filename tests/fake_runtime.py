"""The library on a CUDA runtime without a device (fake_cudart.cpp): what it launches, where and how."""
import ctypes
import os
import subprocess
from collections import namedtuple

import numpy as np

import paper_2603_04359_gb300 as cat
from paper_2603_04359_gb300 import build as catbuild

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(catbuild.__file__), "csrc")
Launch = namedtuple("Launch", "kernel device grid block cluster cooperative arg smem")


def ensure_built():
    """Build the library (and its objects) if it is missing or older than a source."""
    objects = [os.path.join(catbuild.BUILD, os.path.splitext(s)[0] + ".o") for s in catbuild.SOURCES]
    made = [cat.library_path(), *objects]
    newest = max(os.path.getmtime(os.path.join(CSRC, f)) for f in os.listdir(CSRC))
    if not all(os.path.exists(p) for p in made) or newest > min(os.path.getmtime(p) for p in made):
        catbuild.build()
    return objects


class FakeRuntime:
    """The library's entry points over the fake runtime."""

    def __init__(self, folder):
        objects = ensure_built()
        path = os.path.join(str(folder), "libcat_fake.so")
        include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(catbuild.nvcc()))), "include")
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-pthread", "-Wl,-Bsymbolic", "-I", include, "-o", path,
                        os.path.join(HERE, "fake_cudart.cpp"), *objects], check=True, capture_output=True, text=True)
        kept = cat._lib, cat._LIB_PATH
        cat._lib, cat._LIB_PATH = None, path
        try:
            self.lib = cat.load_library()      # the binding's signatures
        finally:
            cat._lib, cat._LIB_PATH = kept
        self.lib.fake_kernel.restype = ctypes.c_char_p
        self.kept = []

    def device(self, d):
        self.lib.fake_set_device(d)

    def record_arg(self, kernel, index):
        self.lib.fake_record_arg(kernel.encode(), index)

    def buffer(self, nbytes=64):
        """Memory the host code may copy from or to, 16-byte aligned."""
        a = np.zeros(nbytes + 16, dtype=np.uint8)
        self.kept.append(a)
        return (a.ctypes.data + 15) & ~15

    def box_rows(self):
        """Rows of the boxes of the last call's tensor maps, in the order they were made."""
        return [self.lib.fake_box_rows(i) for i in range(self.lib.fake_boxes())]

    def call(self, name, *args):
        """The launches of one call, which must succeed; pointers are integers, None is NULL."""
        self.lib.fake_reset()
        status = getattr(self.lib, name)(*args)
        assert status == 0, (name, args, status, self.lib.cat_last_error())
        fields = [[self.lib.fake_field(i, f) for f in range(7)] for i in range(self.lib.fake_launches())]
        return [Launch(self.lib.fake_kernel(i).decode(), *f) for i, f in enumerate(fields)]
