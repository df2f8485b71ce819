"""The library's own sources linked with a CUDA runtime of host memory
(fake_cudart.cpp): its host code runs on a machine without a GPU, with devices,
memory and failing calls as a test wants them. Kernels do nothing."""
import concurrent.futures as cf
import ctypes
import os
import subprocess

import paper_2012_11188_gb300._build as build
from paper_2012_11188_gb300.scan import scan_csr

HERE = os.path.dirname(os.path.abspath(__file__))
HOST, DEVICE = 1, 2  # memory types


class Fake:
    def __init__(self, tmp):
        def run(cmd):
            subprocess.run(cmd, check=True, capture_output=True)

        include = ["-I", os.path.join(build.ROOT, "include")]
        jobs = []
        for src in build.sources():
            obj = os.path.join(tmp, os.path.basename(src) + ".o")
            jobs.append((obj, [build.nvcc(), "-O0", "-Xptxas", "-O0", "-std=c++17", "-Xcompiler",
                               "-fPIC", "--expt-relaxed-constexpr", *build.ARCH, *include, "-c",
                               src, "-o", obj]))
        cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
        obj = os.path.join(tmp, "fake.o")
        jobs.append((obj, ["g++", "-O1", "-std=c++17", "-fPIC", "-I", cuda, "-c",
                           os.path.join(HERE, "fake_cudart.cpp"), "-o", obj]))
        with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 4)) as ex:
            list(ex.map(run, [cmd for _, cmd in jobs]))
        so = os.path.join(tmp, "libscan_fake.so")
        run(["g++", "-shared", "-o", so, *[obj for obj, _ in jobs], "-Wl,-Bsymbolic", "-lpthread"])
        self.lib = ctypes.CDLL(so)
        self.kept = []  # arrays declared as regions stay where they are
        P, Z, I = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_int
        self.lib.fake_log.restype = ctypes.c_char_p
        self.lib.fake_region.argtypes = [P, Z, I, I]
        self.lib.scan_index_build.argtypes = [P, I, P, Z, P]
        self.lib.scan_index_build_batch.argtypes = [P, I, I, P, Z, P]
        self.lib.scan_index_export.argtypes = [P] * 7
        self.lib.scan_index_free.argtypes = [P]
        self.lib.scan_query.argtypes = [P, I, ctypes.c_double, P, I, Z]

    def log(self):
        return self.lib.fake_log().decode().splitlines()

    def region(self, array, kind=DEVICE, device=0, nbytes=None):
        """Declare a numpy array to be memory of a kind and a device (the
        first nbytes of it)."""
        self.kept.append(array)
        self.lib.fake_region(array.ctypes.data, array.nbytes if nbytes is None else nbytes, kind,
                             device)
        return array.ctypes.data

    def csr(self, off, adj, on_device):
        return scan_csr(len(off) - 1, len(adj), off.ctypes.data, off.dtype.itemsize == 8,
                        adj.ctypes.data, on_device)

    def build(self, csr):
        h = ctypes.c_void_p()
        rc = self.lib.scan_index_build(ctypes.byref(csr), 0, None, 0, ctypes.byref(h))
        assert rc == 0, rc
        return h
