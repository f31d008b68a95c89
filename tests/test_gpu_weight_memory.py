"""Table memory of destroyed weights is handed to the next preparation: the results must not depend on that, the amount kept is bounded,
and it goes back to the device with the last object."""
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
    return [t.clone() for g in range(wts.num_groups) for t in wts.view_tensors(g)]

torch.zeros(1, device="cuda")
rot, rot3 = rotation(256, 2), rotation(384, 3)
warm = trdq.trdq_prepare_weights(rot, weight(16, 256, 0), 8)   # kernels loaded, so that free memory only moves with the tables
warm4 = trdq.trdq_prepare_weights(rot, weight(16, 256, 0), 4)
export(warm), export(warm4)
torch.cuda.synchronize()

# the same weights prepared in fresh memory (everything kept alive) and in reused memory, all shapes in both widths
shapes = [(r, n, b) for r in (rot, rot3) for n in (16, 1040, 5008) for b in (8, 4)]
alive = [trdq.trdq_prepare_weights(r, weight(n, r.K, n), b) for r, n, b in shapes]
fresh = [export(w) for w in alive]
del alive
for again in range(3):
    for (r, n, b), want in zip(shapes, fresh):
        w = trdq.trdq_prepare_weights(r, weight(n, r.K, n), b)
        assert all(torch.equal(x, y) for x, y in zip(export(w), want))
        w.close()

# a block that is still read by another stream when its owner is destroyed is not overwritten under that stream
side = torch.cuda.Stream()
a = trdq.trdq_prepare_weights(rot3, weight(5008, 384, 5008), 8)
torch.cuda.synchronize()
with torch.cuda.stream(side):
    torch.cuda._sleep(20_000_000)
    got = a.view_tensors(0)
a.close()
b = trdq.trdq_prepare_weights(rot3, weight(5008, 384, 1), 8)
torch.cuda.synchronize()
assert torch.equal(got[0], fresh[shapes.index((rot3, 5008, 8))][0])
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

# a preparation inside a capture is refused as it is without kept memory, which stays usable
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

# more than the bound is not kept, and the last object gives back everything
big = rotation(4608, 4)
x = weight(16384, 4608, 3)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
w = trdq.trdq_prepare_weights(big, x, 8)
torch.cuda.synchronize()
assert before - torch.cuda.mem_get_info()[0] >= 4 * 16384 * 4608
w.close()
assert torch.cuda.mem_get_info()[0] == before
ws = [trdq.trdq_prepare_weights(rotation(4608, 1), x[:4608].contiguous(), 8) for _ in range(20)]   # 20 x 21 MB
torch.cuda.synchronize()
held = torch.cuda.mem_get_info()[0]
for w in ws:
    w.close()
kept = 20 * 4608 * 4608 - (torch.cuda.mem_get_info()[0] - held)
assert 0 < kept <= 256 << 20, kept
del rot, rot3, big, warm, warm4, w, ws, shapes, a, b, r
gc.collect()
assert torch.cuda.mem_get_info()[0] - held >= 20 * 4608 * 4608, "kept after the last object"
assert trdq.trdq_device_status() == 0
print("ok")
"""


def test_reuse_is_invisible_bounded_and_ends_with_the_last_object():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
