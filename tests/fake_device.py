"""The library's host code on a machine without a GPU: its objects linked with a stand-in CUDA runtime
(fake_cudart.cpp), whose device memory is host memory and whose kernels are recorded and not run."""
from __future__ import annotations

import ctypes
import os
import subprocess

import numpy as np

import paper_1204_0334_gb300 as pkg
from paper_1204_0334_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))
P = ctypes.c_void_p
FLOW = ("W", "P", "blocks", "log_len", "frames", "cn_tiles", "vn_tiles", "nsyn", "N", "sim", "J")


class FakeDevice:
    def __init__(self, folder):
        b.build()
        so = os.path.join(str(folder), "libldpc_fake.so")
        objs = [os.path.join(b.BUILD, os.path.basename(s)[:-3] + ".o") for s in b.sources()]
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "include")
        subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-w", "-I", cuda, "-I", b.CSRC, "-I",
                        os.path.join(b.ROOT, "include"), os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", so],
                       check=True, capture_output=True)
        self.c = ctypes.CDLL(so, mode=os.RTLD_LOCAL | os.RTLD_NOW)
        for name, res, args in pkg._SIGNATURES:
            f = getattr(self.c, name)
            f.restype, f.argtypes = res, args
        self.c.fake_launch_name.restype = ctypes.c_char_p
        self.c.fake_pinned_bytes.restype = ctypes.c_longlong
        self.c.fake_alloc.restype, self.c.fake_alloc.argtypes = P, [ctypes.c_longlong]
        self.c.fake_free.argtypes = [P]
        self.c.fake_budget.argtypes = [ctypes.c_longlong]
        self.keep = []

    def reset(self):
        self.c.fake_reset()
        self.keep.clear()

    def code(self, J, L, p, seed=1):
        import synth

        s = np.ascontiguousarray(synth.qc_shifts(J, L, p, seed=seed), dtype=np.int32)
        h = P()
        assert self.c.ldpc_code_create(s.ctypes.data, J, L, p, ctypes.byref(h)) == 0
        return h

    def device(self, nbytes):
        return P(self.c.fake_alloc(nbytes))

    def calls(self, name):
        return self.c.fake_calls(name.encode())

    def opts(self, **kw):
        return pkg.default_opts(**kw)

    def decode(self, code, N, gamma, *, noalloc=False, post=False, host_out=False, **opts):
        """ldpc_decode (or _noalloc) on device buffers, the decisions to the host with host_out; the status"""
        o = pkg.default_opts(**opts)
        prm = self.device(8 * 256 * o.max_iter) if o.algo == pkg.ALGO_NOMS else None
        o.noms_params = prm
        llr = self.device(4 * gamma * N)
        d_post = self.device(4 * gamma * N) if post else None
        if host_out:
            out = np.zeros(gamma * N, dtype=np.uint8)
            self.keep.append(out)
            hard = P(out.ctypes.data)
        else:
            hard = self.device(gamma * N)
        f = self.c.ldpc_decode_noalloc if noalloc else self.c.ldpc_decode
        st = f(code, llr, gamma, ctypes.byref(o), d_post, hard, None, None, None)
        for x in (prm, llr, d_post, None if host_out else hard):
            if x is not None:
                self.c.fake_free(x)
        return st

    def sim(self, code, frames, slots, target=1 << 60, **opts):
        o = pkg.default_opts(**opts)
        r = pkg.BerResult()
        return self.c.ldpc_ber_sim(code, 2.0, 1, 0, frames, target, slots, ctypes.byref(o), ctypes.byref(r), None)

    def names(self):
        return [self.c.fake_launch_name(i).decode() for i in range(self.c.fake_launches())]

    def flows(self):
        """the launches of the flow decoder, a dict each"""
        out = []
        for i, n in enumerate(self.names()):
            if "tile_kernel" in n and "flow" in n:
                x = (ctypes.c_longlong * len(FLOW))()
                self.c.fake_flow(i, x)
                out.append(dict(zip(FLOW, x)))
        return out
