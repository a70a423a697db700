"""The two update kernels at the edges of their layouts, bit for bit against the
oracle: rows of fewer blocks than a warp has lanes, several warps per row, short
last blocks, every plane count, and the ring kernel of large models (more than
20 M hidden weights)."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle as O
import workloads as W
from paper_2412_00119_gb300 import bmlp as B

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.set_device(DEV)
    O.set_threads(os.cpu_count() or 1)
    B.lib()


def check(widths, h_max, n, bs, p_r0=0.5, gamma=None, group_mode=0):
    gpu = B.BMLP(widths, 7, h_max=h_max, seed=n, bs=bs, p_r0=p_r0, gamma=gamma, group_mode=group_mode)
    ref = O.OracleModel(list(widths), 7, h_max=h_max, seed=n, bs=bs, p_r0=p_r0, gamma=gamma)
    ref.set_group_mode(group_mode)
    xp = W.random_packed(n + 1, n, widths[0])
    y = np.random.default_rng(n).integers(0, 7, n).astype(np.int32)
    x = torch.from_numpy(xp.view(np.int64)).to(DEV)
    e = gpu.train(x, torch.from_numpy(y).to(DEV), count_errors=True)
    assert e == ref.train(W.unpack(xp, widths[0]), y)
    for l in range(1, len(widths)):
        H, Wb, _, p_r, step = gpu.state(l)
        assert np.array_equal(H.astype(np.int32), ref.H(l).T), (widths, l)
        assert np.array_equal(Wb, W.pack(np.where(ref.H(l).T > 0, 1, -1))), (widths, l)
        assert step == ref.step
    gpu.close()


# one block, 1 / 2 / 3 .. 31 / 32 / 33 blocks per row, groups across warps
@pytest.mark.parametrize("h_max", [1, 3, 15, 13, 255, 127, 1001])
@pytest.mark.parametrize("widths", [(1, 5, 40), (64, 37, 65), (130, 64, 33), (2047, 12, 96), (2049, 60, 31),
                                    (4500, 18, 128)])
def test_rows_kernel(widths, h_max):
    check(widths, h_max, 210, 100)


@pytest.mark.parametrize("bs", [1, 127, 129, 300])
def test_rows_kernel_batches(bs):
    check((300, 96, 200), 255, 2 * bs + 1, bs, p_r0=3.0, gamma=[96, 8], group_mode=2)


# short last mini-batches that leave pattern tiles of the forward passes empty, whose
# CTAs have their first weights in flight when they learn it: one tile to all but
# one, with and without a K split
@pytest.mark.parametrize("widths,bs,n", [((70, 200, 130), 100, 101), ((300, 1024, 1024), 100, 117), ((1100, 2100, 257), 64, 65),
                                         ((300, 300, 300, 300), 512, 904), ((2100, 4100, 128), 300, 301)])
def test_empty_pattern_tiles(widths, bs, n):
    check(widths, 255, n, bs)


# more than 20 M weights: the ring kernel, whole rows and ragged ones
@pytest.mark.parametrize("h_max,widths", [(255, (5000, 4500)), (13, (5000, 4500)), (127, (6160, 3600)),
                                          (1001, (2100, 10010))])
def test_ring_kernel(h_max, widths):
    check(widths, h_max, 60, 20)


# steps in a row: the events are drawn beside the first pass or the second
@pytest.mark.parametrize("widths", [(5000, 4500), (4600, 4600, 300)])
def test_ring_kernel_steps(widths):
    check(widths, 255, 18 * 10, 10)


# calls of one mini-batch (their kernels get the inputs as parameters, but for models
# whose draws go beside the later passes), whole and short ones, mixed with a longer
# call and an evaluation
@pytest.mark.parametrize("widths,group_mode,bs", [((70, 40), 0, 16), ((200, 96, 130), 2, 30), ((130, 64, 64, 64), 1, 100),
                                                  ((5000, 4500), 0, 20), ((3000, 4096, 4096), 2, 150), ((300, 8000, 7400), 0, 20)])
def test_calls_of_one_batch(widths, group_mode, bs):
    gpu = B.BMLP(widths, 5, seed=3, bs=bs, group_mode=group_mode)
    ref = O.OracleModel(list(widths), 5, seed=3, bs=bs)
    ref.set_group_mode(group_mode)
    sizes = [bs, bs, max(1, bs // 2), 2 * bs + 1, 1, bs] if widths[0] < 1000 else [bs, 2 * bs, 3]
    n = sum(sizes)
    xp = W.random_packed(5, n, widths[0])
    y = np.random.default_rng(5).integers(0, 5, n).astype(np.int32)
    x, yd, xpm = torch.from_numpy(xp.view(np.int64)).to(DEV), torch.from_numpy(y).to(DEV), W.unpack(xp, widths[0])
    out = torch.empty(n, dtype=torch.int32, device=DEV)
    a = 0
    for m in sizes:
        gpu.train(x[a:a + m], yd[a:a + m])
        gpu.predict(x, out)
        ref.train(xpm[a:a + m], y[a:a + m])
        a += m
    assert np.array_equal(out.cpu().numpy(), ref.predict(xpm))
    for l in range(1, len(widths)):
        H, Wb, _, _, step = gpu.state(l)
        assert np.array_equal(H.astype(np.int32), ref.H(l).T)
        assert np.array_equal(Wb, W.pack(np.where(ref.H(l).T > 0, 1, -1)))
        assert step == ref.step
    gpu.close()


# redrawn groups of a wide model beside a narrower one made after it: in a call of one
# mini-batch, in a longer one, and in both again
def test_group_order_of_two_models():
    widths, bs = (70, 2048, 64), 20
    wide = B.BMLP(widths, 5, seed=9, bs=bs, group_mode=2)
    ref = O.OracleModel(list(widths), 5, seed=9, bs=bs)
    ref.set_group_mode(2)
    narrow = B.BMLP((70, 64), 5, seed=9, bs=bs, group_mode=2)
    sizes = [bs, 3 * bs, bs, 2 * bs]
    xp = W.random_packed(6, sum(sizes), widths[0])
    y = np.random.default_rng(6).integers(0, 5, sum(sizes)).astype(np.int32)
    x, yd, xpm = torch.from_numpy(xp.view(np.int64)).to(DEV), torch.from_numpy(y).to(DEV), W.unpack(xp, widths[0])
    a = 0
    for m in sizes:
        wide.train(x[a:a + m], yd[a:a + m])
        narrow.train(x[a:a + m], yd[a:a + m])
        ref.train(xpm[a:a + m], y[a:a + m])
        a += m
    for l in (1, 2):
        H, _, _, _, step = wide.state(l)
        assert np.array_equal(H.astype(np.int32), ref.H(l).T)
        assert step == ref.step
    wide.close()
    narrow.close()


CAPTURE = """
import ctypes, sys
import numpy as np, torch
import workloads as W
from paper_2412_00119_gb300 import bmlp as B
n, host, count = int(sys.argv[1]), sys.argv[2] == "host", sys.argv[3] == "count"
rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
gpu = B.BMLP((70, 40), 5, seed=3, bs=20)
x, y = W.random_packed(5, n, 70), np.zeros(n, np.int32)
if not host:
    x, y = torch.from_numpy(x.view(np.int64)).cuda(), torch.from_numpy(y).cuda()
gpu.train(x, y)
torch.cuda.synchronize()
s = torch.cuda.Stream()
st, g, nodes = ctypes.c_void_p(s.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
assert rt.cudaStreamBeginCapture(st, 0) == 0
try:
    gpu.train(x, y, count_errors=count, stream=s)
    print("accepted")
except B.BmlpError as e:
    print("refused" if e.code == B.BMLP_ECUDA else e)
# the capture is whole and empty: nothing had gone into the stream
assert rt.cudaStreamEndCapture(st, ctypes.byref(g)) == 0
assert rt.cudaGraphGetNodes(g, None, ctypes.byref(nodes)) == 0
print(nodes.value)
gpu.train(x, y)
print(gpu.state(1)[4] == 2 * -(-n // 20))
"""


# a training call is refused while its stream is captured, before it touches the
# stream, whatever its length, its inputs' place and its results (in a process of its
# own)
@pytest.mark.parametrize("count", ["count", "none"])
@pytest.mark.parametrize("place", ["device", "host"])
@pytest.mark.parametrize("n", [20, 45])
def test_training_is_refused_under_capture(n, place, count):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", CAPTURE, str(n), place, count], cwd=root, capture_output=True, text=True,
                         timeout=300)
    assert run.stdout.split() == ["refused", "0", "True"], run.stdout + run.stderr
