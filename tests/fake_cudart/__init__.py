"""The library on a CUDA runtime without a device (fake_cudart.cpp), for CPU tests of its host side: argument
checks, call order, memory and launches.  Kernels do not run; device pointers are host pointers."""
from __future__ import annotations

import ctypes as ct
import subprocess
from pathlib import Path

import numpy as np

from paper_1807_10633_gb300 import build as B
from paper_1807_10633_gb300 import vmc

CUDA_INCLUDE = Path(B._nvcc()).resolve().parent.parent / "include"


def build(out: Path) -> Path:
    """Link the library's object files with the fake runtime."""
    B.build()
    objs = [B.BUILD / (n + ".o") for n in B.SOURCES]
    if not all(o.exists() for o in objs):
        B.build(force=True)
    lib = out / "libvmc_fake.so"
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", str(CUDA_INCLUDE),
                    str(Path(__file__).parent / "fake_cudart.cpp"), *map(str, objs), "-lgomp", "-o", str(lib)], check=True)
    return lib


class Runtime:
    """The fake runtime's side of the loaded library."""

    def __init__(self, lib: ct.CDLL):
        self.lib = lib
        lib.fake_set.argtypes = [ct.c_uint64, ct.c_int]
        lib.fake_log.restype = ct.c_char_p

    def limit(self, extra: int | None = None, capturing: bool = False):
        """Let at most `extra` more bytes be allocated than are now (None: any number)."""
        self.lib.fake_set(2 ** 63 if extra is None else self.counts()["live"] + extra, int(capturing))

    def counts(self) -> dict:
        out = (ct.c_int64 * 5)()
        self.lib.fake_counts(out)
        return dict(zip(("mallocs", "frees", "uploads", "waits", "live"), out))

    def launches(self) -> list[str]:
        """Names and grids of the kernels launched since the last call, in order."""
        log = self.lib.fake_log().decode().split("\n")[:-1]
        self.lib.fake_clear()
        return log


class System:
    """Lists and W walkers of one system on a context; arrays on the host, `shift` bytes off a 256-byte boundary."""

    def __init__(self, ctx, system, W: int, eps: float, precision: int = vmc.VMC_MIXED, shift: dict | None = None):
        self.ctx, self.eps, self.W = ctx, float(eps), W
        self.lists = vmc.vmc_build_screened_lists(ctx, system.M, system.h1, system.eri, system.e_core, eps)
        n = vmc.vmc_walkers_sizes(W, system.M, system.n_alpha, system.n_beta, self.lists)
        real = 8 if precision == vmc.VMC_FP64 else 4
        names = ("occ_bits", "occ_list", "virt_list", "pos", "G", "AinvT", "S", "F", "e_diag", "rng_counter")
        self._keep, ptr = [], {}
        for name, k, size in zip(names, n, (4, 2, 2, 2, real, real, real, real, 8, 8)):
            ptr[name] = self._array(k * size, (shift or {}).get(name, 0))
        N2 = 2 * system.M
        J, Ca, Cb = (self._array(8 * k) for k in (N2 * N2, system.M * system.n_alpha, system.M * system.n_beta))
        self.params = vmc.vmc_params(J, Ca, Cb, None, None)
        self.walkers = vmc.vmc_walkers(W, system.M, system.n_alpha, system.n_beta, precision, *(ptr[k] for k in names), None)
        self.e, self.t, self.codes = (self._array(8 * W) for _ in range(3))
        vmc.vmc_walkers_init(ctx, self.lists, self.params, self.walkers)

    def _array(self, n_bytes: int, shift: int = 0) -> int:
        a = np.zeros(n_bytes + 512, dtype=np.uint8)
        self._keep.append(a)
        return (a.ctypes.data + 255) // 256 * 256 + shift

    def energy(self, eps_run: float | None = None, ctx=None):
        vmc.vmc_local_energy(ctx or self.ctx, self.lists, self.params, self.walkers,
                             self.eps if eps_run is None else eps_run, self.e, self.t)

    def step(self, lists=None):
        vmc.vmc_ctmc_step(self.ctx, lists or self.lists, self.params, self.walkers, 3, self.codes)

    def close(self):
        vmc.vmc_lists_destroy(self.lists)


def batch(systems):
    """Batch items over several systems of one context (the caller keeps the systems)."""
    items = (vmc.vmc_batch_item * len(systems))()
    for it, s in zip(items, systems):
        it.lists, it.params, it.walkers = s.lists, ct.pointer(s.params), ct.pointer(s.walkers)
        it.eps_run, it.d_e_loc, it.d_t_res, it.d_move_code = s.eps, s.e, s.t, s.codes
    return items
