"""The library's own host code (every .cu file of the package) linked against a CUDA runtime that has no device
(tests/fake_cudart.cpp): for tests of what a call asks of the runtime and enqueues, on the CPU."""
import ctypes as C
import os
import re
import subprocess
from collections import namedtuple

from paper_2510_20707_b200 import binding, build

Launch = namedtuple("Launch", "caller grid threads cluster kernel")


class FakeCuda:
    """`lib` as binding.load_library() gives it; `runtime` the functions of fake_cudart.cpp."""

    def __init__(self, directory):
        path = os.path.join(directory, "libmixkv_fake.so")
        src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fake_cudart.cpp")
        subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_100a,code=compute_100a", "-O1",
                        "-std=c++17", "--threads", "0", "-Xcompiler", "-fPIC", "-shared", "-cudart", "none", "-Xlinker",
                        "-Bsymbolic", f"-I{build.INCLUDE}", f"-I{build.CSRC}", "-o", path, src, *build.sources()],
                       check=True)
        self.runtime = C.CDLL(path)
        self.runtime.fake_launch.restype = C.c_char_p
        kept = binding.LIB_PATH, binding._lib
        binding.LIB_PATH, binding._lib = path, None
        try:
            self.lib = binding.load_library()
        finally:
            binding.LIB_PATH, binding._lib = kept
        self.reset()

    def reset(self, device=0, sms=148, major=10, query_error=0, ask_error=0, pause_us=0, resident={}):
        """What the library keeps per device it keeps by its number: a test that changes the answers takes another."""
        self.runtime.fake_reset(device, sms, major, query_error, ask_error, pause_us)
        for size, clusters in resident.items():
            self.runtime.fake_resident(size, clusters)

    def launches(self):
        out = []
        for i in range(self.runtime.fake_launches()):
            v = [C.c_int() for _ in range(4)]
            name = self.runtime.fake_launch(i, *[C.byref(x) for x in v]).decode()
            out.append(Launch(*[x.value for x in v], re.search(r"k_[a-z0-9_]+", name).group(0).split("IL")[0]))
        return out

    def last_error(self):
        return self.runtime.cudaPeekAtLastError()
