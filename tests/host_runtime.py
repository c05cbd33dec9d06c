"""The library linked to the stand-in runtime of tests/host/fake_cudart.cpp:
its host code (allocation, uploads, launches) runs here without a GPU.  The
tests run each scenario in a process of its own, because the library keeps
what it has asked of a device."""
import ctypes as C
import os
import subprocess
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def build_library(out_dir) -> str:
    """libcsph's objects and the stand-in runtime as one shared library."""
    from paper_1805_05128_gb300 import build
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    so = os.path.join(str(out_dir), "libcsph_host.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-Wl,-Bsymbolic", "-I", "/usr/local/cuda/include",
                    os.path.join(ROOT, "tests", "host", "fake_cudart.cpp"), *objs, "-o", so, "-lpthread"], check=True)
    return so


def run(so: str, scenario: str, *args) -> str:
    """A scenario (a function of the module named in `scenario`) in a fresh process."""
    module, func = scenario.split(":")
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([ROOT, os.path.join(ROOT, "tests")]))
    code = f"import sys, {module} as m; print(m.{func}(sys.argv[1], *map(int, sys.argv[2:])))"
    r = subprocess.run([sys.executable, "-c", code, so, *map(str, args)], capture_output=True, text=True, timeout=300, env=env)
    assert r.returncode == 0, f"exit {r.returncode}\n{r.stdout}\n{r.stderr}"
    return r.stdout.strip()


class Host:
    """Handles of a lattice gas whose arrays are host memory."""

    def __init__(self, so: str):
        from paper_1805_05128_gb300 import abi
        abi.SO_PATH = so
        self.abi, self.L = abi, abi.lib()
        self.L.fake_launches.restype = C.c_char_p
        self.L.fake_copied.restype = self.L.fake_changed.restype = C.c_longlong
        self.keep = []

    def array(self, n, dtype=np.float64):
        a = np.ones(n, dtype=dtype)
        self.keep.append(a)
        return a

    def state(self, n):
        abi, s = self.abi, self.abi.sph_state()
        s.n = n
        for k in abi.STATE_F64 + abi.STATE_RATES + abi.STATE_DERIVED:
            setattr(s, k, self.array(n).ctypes.data)
        s.unit = self.array(n, np.int32).ctypes.data
        return s

    def handle(self, state, offsets=None, **params):
        abi, p = self.abi, self.abi.sph_params()
        p.dim, p.kernel, p.precision, p.n_mat = 3, abi.SPH_KERNEL_CUBIC, abi.SPH_PREC_MIXED, 1
        p.kappa, p.eta, p.cfl, p.cell_cap = 2.0, 1.3, 0.3, 1 << 16
        p.mat[0].eos, p.mat[0].gamma = abi.SPH_EOS_IDEAL, 1.4
        for k, v in params.items():
            setattr(p, k, v)
        return abi.sph_init(p, len(offsets or [0, 1]) - 1, offsets or [0, state.n], state, 0)

    def launches(self):
        """(kernel name, blocks, CTAs a cluster) of every launch since the last call."""
        rows = [r.split() for r in self.L.fake_launches().decode().splitlines()]
        self.L.fake_clear()
        return [(r[0], int(r[1]), int(r[2])) for r in rows]
