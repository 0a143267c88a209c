"""The library's host code on a stand-in for the CUDA runtime (fake_cudart.cpp): which kernels a
call launches, with what shapes and memory, and what it does when a call fails.

Kernels are named as in the sources with their template arguments, e.g.
``mh_spec_kernel<2,4,0>``; they are not run.
"""
import ctypes as ct
import glob
import importlib.util
import os
import re
import subprocess
from unittest import mock

from paper_2511_22094_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
OOM = 2  # cudaErrorMemoryAllocation
HOOK = ct.CFUNCTYPE(ct.c_int, ct.c_char_p, ct.c_char_p, ct.POINTER(ct.c_longlong), ct.POINTER(ct.c_void_p))

#: resident blocks an SM that the kernels' registers allow (launch bounds; shared memory on top)
RESIDENT = [(r"mh(_slice)?_kernel<(2|4),", 2), (r"mh(_slice)?_kernel<3,", 4), (r"mh_kernel", 4), (r"mh_spec_kernel<\d,2,", 2),
            (r"mh_split|mh_spec", 1), (r"fit_many_kernel<\d+,1", 20), (r"fit_(step|list)_kernel<\d+,1", 5), (r"", 2)]


def short(mangled):
    """``_ZN3gac9mh_kernelILi2ELi0ELb0ELi256EEEv...`` -> ``mh_kernel<2,0,0,256>``."""
    m = re.search(r"\d([a-z_]+_kernel)(I((?:L[ibx]\d+E|[fd])+)E)?", mangled)
    if not m:
        return mangled
    args = [a or b for a, b in re.findall(r"L[ibx](\d+)E|([fd])", m.group(3) or "")]
    if m.group(1) == "mh_kernel":  # the form: 3 where it is the short protocols' own
        args[4:] = ["short"] * (args[4] == "3")
    return m.group(1) + (f"<{','.join(args)}>" if args else "")


class FakeGpu:
    """Records launches (name, grid x, grid y, block, shared bytes) and settings; `memory` bounds the
    device memory in use; `on_launch(name, args)` may return an error code; `on_limit(name)` runs when
    a call has set a kernel's shared-memory limit."""

    def __init__(self, lib):
        self.lib = lib
        self.hook = HOOK(self._call)
        lib.fake_set_hook(self.hook)
        self.reset()

    def reset(self):
        self.launches, self.limits, self.sizes = [], [], []
        self.in_use = self.peak = 0
        self.memory = None
        self.on_launch = self.on_limit = None
        self.lib.fake_forget_limits()

    def _call(self, op, kernel, x, args):
        name = short(kernel.decode())
        if op == b"malloc":
            self.sizes.append(x[0])
            if self.memory is not None and self.in_use + x[0] > self.memory:
                return OOM
            self.in_use += x[0]
            self.peak = max(self.peak, self.in_use)
        elif op == b"free":
            self.in_use -= x[0]
        elif op == b"attr" and x[0] == 8:  # MaxDynamicSharedMemorySize
            self.limits.append((name, x[1]))
            if self.on_limit:
                self.on_limit(name)
        elif op == b"occupancy":
            block, smem = x[0], x[1]
            by_regs = next(n for pat, n in RESIDENT if re.search(pat, name)) * (1 if "fit_" in name or "mh_s" in name else 256 // block)
            return min(by_regs, 2048 // block, 228 * 1024 // (smem + 2048))
        elif op == b"launch":
            self.launches.append((name, x[0], x[1], x[2], x[3]))
            if self.on_launch:
                return self.on_launch(name, args) or 0
        return 0

    def names(self):
        return [n for n, *_ in self.launches]

    def device(self, *arrays):
        """Lets the library take these numpy arrays for device memory (until `host`)."""
        for a in arrays:
            self.lib.fake_mark_device(ct.c_void_p(a.ctypes.data), 1)

    def host(self, *arrays):
        for a in arrays:
            self.lib.fake_mark_device(ct.c_void_p(a.ctypes.data), 0)


def load(tmp_path):
    """(binding module, FakeGpu) on a build of the library's objects with the stand-in."""
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in sorted(glob.glob(os.path.join(build.CSRC, "*.cu")))]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    path = os.path.join(str(tmp_path), "libgac_fake.so")
    subprocess.run([build._nvcc(), "-std=c++17", "-O1", "-cudart", "none", "-shared", "-Xcompiler", "-fPIC", "-Xlinker", "-Bsymbolic", "-o", path,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-lpthread"], check=True, capture_output=True)
    real = ct.CDLL
    spec = importlib.util.spec_from_file_location("gac_on_fake_gpu", os.path.join(build.PKG, "gac.py"))
    mod = importlib.util.module_from_spec(spec)
    with mock.patch.object(ct, "CDLL", lambda p: real(path)):
        spec.loader.exec_module(mod)
    return mod, FakeGpu(mod.lib())
