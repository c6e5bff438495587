"""The library linked against a runtime that only writes down what it is asked to
queue (tests/c/fake_cudart.c), so that the host side of a call can be tested
without a GPU: which kernels, how many CTAs, behind which copies."""
from __future__ import annotations

import ctypes
import os
import re
import subprocess
import tempfile

import pytest

from paper_0912_0947_gb300 import build as B

HERE = os.path.dirname(os.path.abspath(__file__))
_vp, _u64, _u32 = ctypes.c_void_p, ctypes.c_uint64, ctypes.c_uint32


class Launches:
    """Calls on made-up device addresses (nothing is read or written there)."""

    def __init__(self):
        try:
            nvcc = B.nvcc()
        except RuntimeError:
            pytest.skip("nvcc not available")
        objs = [os.path.join(B.BUILD, os.path.basename(p)[:-3] + ".o") for p in B.sources()]
        B.build(force=not all(map(os.path.exists, objs)))
        self.dir = tempfile.TemporaryDirectory()
        fake = os.path.join(self.dir.name, "fake.o")
        so = os.path.join(self.dir.name, "libstego_launches.so")
        cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
        subprocess.run(["gcc", "-O1", "-fPIC", "-I" + cuda, "-c", os.path.join(HERE, "c", "fake_cudart.c"),
                        "-o", fake], check=True)
        subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,--no-undefined", "-o", so,
                        *objs, fake, "-lpthread", "-ldl"],
                       check=True)
        self.lib = ctypes.CDLL(so)
        self.lib.fake_log.restype = ctypes.c_char_p
        self.lib.stego_embed.argtypes = [_vp, _vp, _u64, _vp, _u64, _vp, _u32, _vp, _vp]
        self.lib.stego_extract.argtypes = [_vp, _u64, _vp, _u64, _u64, _vp, _u32, _vp, _vp]
        self.lib.stego_changed_bytes.argtypes = [_vp, _vp, _u64, _vp, _vp]

    def queued(self, name, *args, capturing=False):
        """The call's queue: ("memset", bytes) and (kernel, grid, block, programmatic)."""
        self.lib.fake_reset(int(capturing))
        assert getattr(self.lib, name)(*args) == 0
        out = []
        for line in self.lib.fake_log().decode().splitlines():
            if line.startswith("memset"):
                out.append(("memset", int(line.split()[1])))
            else:
                m = re.fullmatch(r"launch (\S+) grid=(\d+) block=(\d+) programmatic=(\d)", line)
                out.append((m[1], int(m[2]), int(m[3]), int(m[4])))
        return out

    @property
    def wave(self):
        """CTAs that are resident together."""
        return self.lib.fake_wave()
