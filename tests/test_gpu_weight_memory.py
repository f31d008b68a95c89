"""Weights own their device memory: what an object computes does not depend on what its memory held before, and destroying it returns all of
the memory to the device at once, whatever else is alive."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import gc
import threading
import numpy as np
import torch
from paper_2503_06564_b200 import trdq

def rotation(K, G):
    rng = np.random.default_rng(K + G)
    return trdq.Rotation(K, np.linspace(0, 1000, G + 1).astype(np.int32), (rng.integers(0, 2, (G, K)) * 2 - 1).astype(np.int8), None)

def weight(N, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn((N, K), generator=g, device="cuda") * 0.02).to(torch.bfloat16)

def export(wts):
    # all tables of a weights object: codes and scales as they are, column sums and 4-bit multipliers through the products that use them
    out = [t.clone() for g in range(wts.num_groups) for t in wts.view_tensors(g)]
    g = torch.Generator(device="cuda").manual_seed(wts.K)
    codes = torch.randint(-127, 128, (37, wts.K), generator=g, device="cuda", dtype=torch.int8)
    scales = torch.rand((37,), generator=g, device="cuda")
    zero = torch.randint(0, 256, (37,), generator=g, device="cuda", dtype=torch.int32)
    for i in range(wts.num_groups):
        t = i * 1000 // wts.num_groups + 1
        out.append(trdq.trdq_linear(wts, t, codes, scales))
        if wts.wbits == 8:
            out.append(trdq.trdq_linear_asym(wts, t, codes.view(torch.uint8), scales, zero))
    return [t.view(torch.uint8) for t in out]

torch.zeros(1, device="cuda")
rot, rot3 = rotation(256, 2), rotation(384, 3)
warm = trdq.trdq_prepare_weights(rot, weight(16, 256, 0), 8)   # kernels loaded, so that free memory only moves with the tables
warm4 = trdq.trdq_prepare_weights(rot, weight(16, 256, 0), 4)
export(warm), export(warm4)
torch.cuda.synchronize()

# the same weights prepared with everything kept alive and after others were destroyed, all shapes in both widths
shapes = [(r, n, b) for r in (rot, rot3) for n in (16, 1040, 5008) for b in (8, 4)]
alive = [trdq.trdq_prepare_weights(r, weight(n, r.K, n), b) for r, n, b in shapes]
fresh = [export(w) for w in alive]
del alive
for again in range(3):
    for (r, n, b), want in zip(shapes, fresh):
        w = trdq.trdq_prepare_weights(r, weight(n, r.K, n), b)
        assert all(torch.equal(x, y) for x, y in zip(export(w), want))
        w.close()

# memory that is still read by another stream when its owner is destroyed is not overwritten under that stream
side = torch.cuda.Stream()
a = trdq.trdq_prepare_weights(rot3, weight(5008, 384, 5008), 8)
torch.cuda.synchronize()
with torch.cuda.stream(side):
    torch.cuda._sleep(20_000_000)
    got = a.view_tensors(0)
a.close()
b = trdq.trdq_prepare_weights(rot3, weight(5008, 384, 1), 8)
torch.cuda.synchronize()
assert torch.equal(got[0].view(torch.uint8), fresh[shapes.index((rot3, 5008, 8))][0])
b.close()

# several threads, each on its own stream
def work(i, failed):
    with torch.cuda.stream(torch.cuda.Stream()):
        for j in range(8):
            k = (3 * i + j) % len(shapes)
            r, n, bits = shapes[k]
            x = weight(n, r.K, n)
            w = trdq.trdq_prepare_weights(r, x, bits)
            out = export(w)
            torch.cuda.current_stream().synchronize()
            if not all(torch.equal(p, q) for p, q in zip(out, fresh[k])):
                failed.append((i, j))
            w.close()
failed = []
threads = [threading.Thread(target=work, args=(i, failed)) for i in range(4)]
[t.start() for t in threads]
[t.join() for t in threads]
assert not failed, failed

# a preparation inside a capture is refused
x = weight(1040, 256, 1040)
graph = torch.cuda.CUDAGraph()
try:
    with torch.cuda.graph(graph):
        trdq.trdq_prepare_weights(rot, x, 8)
    raise SystemExit("a preparation was captured")
except (trdq.TrdqError, RuntimeError):
    pass
torch.cuda.synchronize()

# another thread may destroy weights while this one captures (thread-local mode), and the capture holds
w = trdq.trdq_prepare_weights(rot, x, 8)
y = torch.zeros(1024, device="cuda")
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, capture_error_mode="thread_local"):
    y += 1.0
    t = threading.Thread(target=w.close)
    t.start()
    t.join()
    y += 1.0
graph.replay()
torch.cuda.synchronize()
assert float(y.sum()) == 2048.0

# objects destroyed by a thread that captures: the capture is lost, the next calls are not
for bits in (8, 4):
    for obj in (trdq.trdq_prepare_weights(rot, x, bits), rotation(256, 2)):
        torch.cuda.synchronize()
        try:
            with torch.cuda.graph(torch.cuda.CUDAGraph(), capture_error_mode="thread_local"):
                obj.close()
            raise SystemExit("memory was freed inside a capture")
        except RuntimeError:
            pass
        torch.cuda.synchronize()
        trdq.trdq_prepare_weights(rot, x, bits).close()

# everything is returned at once, with rotations and other weights alive: another allocator may want it
big = [rotation(4608, 4), rotation(4608, 1)]
x = weight(16384, 4608, 3)
small = x[:4608].contiguous()
for r, m, bits in ((big[0], x, 8), (big[1], small, 8), (big[1], small, 4)):
    trdq.trdq_prepare_weights(r, m, bits).close()   # kernels loaded
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
w = trdq.trdq_prepare_weights(big[0], x, 8)
torch.cuda.synchronize()
assert before - torch.cuda.mem_get_info()[0] >= 4 * 16384 * 4608
w.close()
assert torch.cuda.mem_get_info()[0] == before, torch.cuda.mem_get_info()[0] - before
ws = [trdq.trdq_prepare_weights(big[1], small, bits) for bits in (8, 4) for _ in range(10)]
torch.cuda.synchronize()
held = torch.cuda.mem_get_info()[0]
for w in ws:
    w.close()
assert torch.cuda.mem_get_info()[0] - held >= 10 * 4608 * 4608 * 3 // 2, torch.cuda.mem_get_info()[0] - held
assert trdq.trdq_device_status() == 0
print("ok")
"""


def test_tables_are_the_objects_own_and_go_back_with_it():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
