"""A new run's control block: init_ctl, compiled for the host, must set every byte of it
(the one-launch runs of small graphs start from uninitialised shared memory and copy the
whole block back), whatever it held before."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cstring>
#include "ss_device.cuh"
extern "C" int init_block(unsigned char fill, unsigned char* out) {
  int rdeg[1] = {7};
  ss_iter_stats iters[1];
  ss::Dev d;
  std::memset(&d, 0, sizeof d);
  d.n = 1;
  d.rdeg = rdeg;
  d.iters = iters;
  std::memset(out, fill, sizeof(ss::Ctl));
  ss::init_ctl(d, reinterpret_cast<ss::Ctl*>(out), 0);
  return (int)sizeof(ss::Ctl);
}
"""


def test_init_sets_every_byte(tmp_path):
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("no nvcc")
    src, lib = tmp_path / "block.cu", tmp_path / "block.so"
    src.write_text(SRC)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_2010_09913_gb300", "csrc"),
                    str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).init_block
    blocks = []
    for fill in (0x00, 0xA5):
        out = (ctypes.c_ubyte * 4096)()
        size = f(ctypes.c_ubyte(fill), out)
        blocks.append(np.frombuffer(out, np.uint8)[:size].copy())
    np.testing.assert_array_equal(blocks[0], blocks[1])
