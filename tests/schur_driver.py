"""Builds schur_driver.cu against the library and converts fields: the passes of
the even-odd stencil (csrc/schur.cu) for the tests, which the C ABI reaches only
inside whole solves."""
import ctypes as C
import os
import subprocess

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))


def load(m, tmp):
    import torch
    from paper_2412_06347_gb300 import build as b
    so = os.path.join(str(tmp), "schur_driver.so")
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-shared", os.path.join(HERE, "schur_driver.cu"), b.LIB, "-o", so,
                    "-Xlinker", "-rpath=" + os.path.dirname(b.LIB)], check=True, capture_output=True)
    lib = C.CDLL(so)

    def call(name, ctx, g, *args):
        conv = [C.c_void_p(a.data_ptr()) if hasattr(a, "data_ptr") else C.c_void_p() if a is None else C.c_int(a)
                for a in args]
        torch.cuda.synchronize()  # the context's stream does not wait for torch's
        st = getattr(lib, "drv_" + name)(ctx.handle, C.c_void_p(g), *conv)
        assert st == 0, (name, st, m.mglma_last_error())

    def ready(ctx, g):
        u = C.c_int()
        assert lib.drv_ready(ctx.handle, C.c_void_p(g), C.byref(u)) == 0
        return bool(u.value)

    call.ready = ready
    return call


def parity_sites(L):
    """(even sites, odd sites) in site order: entry u is the site of half-lattice index u."""
    p = np.indices(L).sum(axis=0).reshape(-1) % 2
    return np.flatnonzero(p == 0), np.flatnonzero(p == 1)


def to_half(psi, sites, dtype):
    """Canonical spinors (n, L..., 4, 3), the given parity, as a device half field."""
    import torch
    n = psi.shape[0]
    v = np.ascontiguousarray(psi.reshape(n, -1, 12)[:, sites].transpose(0, 2, 1))  # n, 12, Vh
    r = np.stack([v.real, v.imag], -1).astype(np.float32)
    per = 2 if dtype == torch.float32 else 4  # complex components per 16 bytes
    r = r.reshape(n, 12 // per, per, len(sites), 2).transpose(0, 1, 3, 2, 4).reshape(n, 12 // per, len(sites), 2 * per)
    return torch.from_numpy(np.ascontiguousarray(r)).cuda().to(dtype)


def from_half(t):
    """A device half field as complex128 (n, Vh, 12)."""
    n, rows, Vh, reals = t.shape
    r = t.to("cpu").double().numpy().reshape(n, rows, Vh, reals // 2, 2).transpose(0, 2, 1, 3, 4).reshape(n, Vh, 12, 2)
    return r[..., 0] + 1j * r[..., 1]
