"""GPU test: the native calls allocate their outputs and workspaces without the GIL, so that other Python threads run while torch's allocator waits."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# An allocator for a memory pool that hands out pieces of one tensor's memory and notes whether its caller held the GIL.
ALLOCATOR = """
#include <cstddef>
#include <sys/types.h>
extern "C" {
int PyGILState_Check(void);
static char* next;
static size_t left;
static int asked, held;
void lend(char* p, size_t n) { next = p; left = n; }
void* take(ssize_t n, int, void*) {
  const size_t size = (static_cast<size_t>(n) + 511) / 512 * 512;
  ++asked;
  held += PyGILState_Check();
  if (size > left) return nullptr;
  char* const p = next;
  next += size;
  left -= size;
  return p;
}
void give(void*, ssize_t, int, void*) {}
void counts(int* a, int* h) { *a = asked; *h = held; asked = held = 0; }
}
"""


def test_outputs_are_allocated_without_the_gil(tmp_path):
    import torch
    from paper_2503_06564_b200 import trdq
    source, built = tmp_path / "allocator.cpp", str(tmp_path / "allocator.so")
    source.write_text(ALLOCATOR)
    subprocess.run([os.environ.get("CXX", "g++"), "-std=c++17", "-shared", "-fPIC", str(source), "-o", built], check=True)
    c = ctypes.CDLL(built)
    slab = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
    skip = 1 << 20   # torch's allocator knows blocks by their first byte, and the tensor is one
    c.lend(ctypes.c_void_p(slab.data_ptr() + skip), ctypes.c_size_t(slab.numel() - skip))
    allocator = torch.cuda.memory.CUDAPluggableAllocator(built, "take", "give")

    M, N, K = 16, 32, 8192
    rot = trdq.Rotation(K, [0, 1000], np.ones((1, K), np.int8), None)
    x = torch.randn((M, K), device="cuda").bfloat16()
    wts = trdq.trdq_prepare_weights(rot, torch.randn((N, K), device="cuda").bfloat16(), 8)
    codes, scales = trdq.trdq_rotate_quantize(rot, 0, x)
    u8, su, zp = trdq.trdq_rotate_quantize_asym(rot, 0, x)
    y = trdq.trdq_linear(wts, 0, codes, scales)
    assert trdq.trdq_linear_splitk_workspace(wts, M)[1] > 0
    for call in (lambda: trdq.trdq_rotate_quantize(rot, 0, x), lambda: trdq.trdq_norm_rotate_quantize(rot, 0, x), lambda: trdq.trdq_rotate_quantize_asym(rot, 0, x),
                 lambda: trdq.trdq_linear(wts, 0, codes, scales), lambda: trdq.trdq_linear_act(wts, 0, codes, scales), lambda: trdq.trdq_linear_asym(wts, 0, u8, su, zp),
                 lambda: trdq.trdq_linear_cfg(wts, 0, [codes, codes], [scales, scales]), lambda: trdq.trdq_linear_splitk(wts, 0, codes, scales),
                 lambda: trdq.trdq_linear_splitk(wts, 0, codes, scales, None, y)):
        pool = torch.cuda.MemPool(allocator.allocator())
        with torch.cuda.use_mem_pool(pool):
            out = call()
        torch.cuda.synchronize()
        asked, held = ctypes.c_int(), ctypes.c_int()
        c.counts(ctypes.byref(asked), ctypes.byref(held))
        assert asked.value > 0 and held.value == 0
        del out, pool
    assert trdq.trdq_device_status() == 0
