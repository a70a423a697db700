"""The evaluation and front-end kernels at the edges of their tiles (MMA tiles,
K pieces, K splits, odd word counts, single rows), bit for bit against the
oracle."""
import os

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


def dev(xp):
    return torch.from_numpy(np.ascontiguousarray(xp).view(np.int64)).to(DEV)


# widths K, N and patterns n: tiles of 128 neurons and 16 .. 112 patterns, pieces
# of 1024 and k-steps of 256 inputs, splits of 1 .. 4, rows of odd word counts
SMALL = [(1, 1, 1), (63, 127, 15), (64, 128, 16), (255, 129, 17), (257, 300, 112), (784, 1024, 100),
         (1000, 525, 113), (1023, 130, 33), (1025, 640, 100), (2049, 70, 7), (3072, 4096, 128),
         (5000, 257, 200), (8190, 1000, 100), (32767, 33, 9), (960, 8192, 512)]


@pytest.mark.parametrize("K,N,n", SMALL)
def test_small_batch_forward(K, N, n):
    gpu = B.BMLP((K, N), 4, seed=K + N, bs=64)
    ref = O.OracleModel([K, N], 4, seed=K + N, bs=64)
    xp = W.random_packed(n, n, K)
    _, a = O.layer_forward(W.unpack(xp, K), ref.H(1))
    want = W.pack(a)
    out = torch.full((n, W.words(N)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_layer_forward(gpu.h, 1, dev(xp), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), want)
    # rows that start 8 bytes off a 16-byte boundary, with pad bits set
    xp2 = np.zeros(n * W.words(K) + 1, np.uint64)
    rows = xp2[1:].reshape(n, -1)
    rows[:] = xp
    if K % 64:
        rows[:, -1] |= ~np.uint64((1 << (K % 64)) - 1)
    x2 = dev(xp2)[1:].view(n, -1)
    out.fill_(-1)
    B.bmlp_layer_forward(gpu.h, 1, x2, out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), want)
    gpu.close()


# more patterns: several pattern tiles, most of them still too few for the pairs
LARGE = [(1, 1, 513), (255, 255, 700), (784, 257, 1300), (1000, 525, 2000), (2049, 300, 1025),
         (4096, 512, 900), (32767, 33, 600), (64, 2048, 11000)]


@pytest.mark.parametrize("K,N,n", LARGE)
def test_large_batch_forward(K, N, n):
    gpu = B.BMLP((K, N), 4, seed=K + N, bs=64)
    ref = O.OracleModel([K, N], 4, seed=K + N, bs=64)
    xp = W.random_packed(n, n, K)
    _, a = O.layer_forward(W.unpack(xp, K), ref.H(1))
    out = torch.full((n, W.words(N)), -1, dtype=torch.int64, device=DEV)
    x2 = np.array(xp)
    if K % 64:
        x2[:, -1] |= ~np.uint64((1 << (K % 64)) - 1)   # pad bits set: ignored
    B.bmlp_layer_forward(gpu.h, 1, dev(x2), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), W.pack(a))
    gpu.close()


# pairs of CTAs on 256 x 256 tiles, several tiles per pair: ragged neuron tiles (one
# CTA of a pair short or empty), rows and outputs of odd word counts, one to 32 pieces
# of K, a short last pattern tile
PAIRS = [(1000, 255, 20000), (1000, 525, 4096), (1060, 130, 10007), (2049, 300, 12000), (5000, 257, 9000), (32767, 33, 3000),
         (960, 640, 5000)]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("K,N,n", PAIRS)
def test_pair_forward(K, N, n, off):
    # (the dispatch takes the small tiles while they fit the SMs once and their
    # pieces 1.6 times)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-n // 112) * -(-N // 128)
    assert tiles > sms or 5 * tiles * -(-K // 1024) > 8 * sms
    gpu = B.BMLP((K, N), 4, seed=K + N, bs=64)
    ref = O.OracleModel([K, N], 4, seed=K + N, bs=64)
    xp = W.random_packed(n, n, K)
    _, a = O.layer_forward(W.unpack(xp, K), ref.H(1))
    # rows from a word's offset on, pad bits set (ignored), the output's neighbours kept
    buf = np.zeros(n * W.words(K) + off, np.uint64)
    rows = buf[off:].reshape(n, -1)
    rows[:] = xp
    if K % 64:
        rows[:, -1] |= ~np.uint64((1 << (K % 64)) - 1)
    out = torch.full((n * W.words(N) + off + 2,), -1, dtype=torch.int64, device=DEV)
    B.bmlp_layer_forward(gpu.h, 1, dev(buf)[off:].view(n, -1), out[off:-2].view(n, -1))
    assert np.array_equal(out[off:-2].view(n, -1).cpu().numpy().view(np.uint64), W.pack(a))
    assert (out[:off] == -1).all() and (out[-2:] == -1).all()
    gpu.close()


# evaluation captured into a graph right behind a memset, a copy and a kernel of another
# library that write its input, and replayed on other inputs
@pytest.mark.parametrize("before", ["memset", "copy", "kernel"])
@pytest.mark.parametrize("n", [100, 20000])
def test_evaluation_in_a_graph(n, before):
    widths = [300, 257, 130]
    gpu = B.BMLP(widths, 10, seed=n, bs=64)
    src = dev(W.random_packed(n, n, widths[0]))
    x = src.clone()
    last, every = (torch.empty(s, dtype=torch.int32, device=DEV) for s in ((n,), (2, n)))
    layer = torch.empty((n, W.words(widths[1])), dtype=torch.int64, device=DEV)

    def write():
        if before == "memset":
            x.zero_()
        elif before == "copy":
            x.copy_(src)
        else:
            torch.bitwise_not(src, out=x)

    def calls():
        write()
        gpu.predict(x, last)
        write()
        gpu.predict_layers(x, every)
        write()
        B.bmlp_layer_forward(gpu.h, 1, x, layer)

    calls()   # allocates the scratch
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        calls()
    for seed in (1, 2):
        src.copy_(dev(W.random_packed(seed, n, widths[0])))
        calls()
        want = [t.clone() for t in (last, every, layer)]
        for t in (last, every, layer, x):
            t.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(t, w) for t, w in zip((last, every, layer), want))
    gpu.close()


@pytest.mark.parametrize("classes", [2, 33, 100, 128, 129])
@pytest.mark.parametrize("n", [1, 113, 700])
def test_labels_of_every_layer(classes, n):
    widths = [300, 257, 1030]
    gpu = B.BMLP(widths, classes, seed=classes, bs=64)
    ref = O.OracleModel(widths, classes, seed=classes, bs=64)
    xp = W.random_packed(7 * n, n, widths[0])
    x = W.unpack(xp, widths[0])
    out = torch.full((2, n), -1, dtype=torch.int32, device=DEV)
    gpu.predict_layers(dev(xp), out)
    assert np.array_equal(out.cpu().numpy(), ref.predict_layers(x))
    last = torch.full((n,), -1, dtype=torch.int32, device=DEV)
    gpu.predict(dev(xp), last)
    assert np.array_equal(last.cpu().numpy(), ref.predict(x))
    gpu.close()


# chunks of 64 inputs, blocks of 256, neuron tiles of 64 to 256 in steps of 32, the widest
# tensor-core shape (4608) and the first past it, rows that allow copies of 16,
# 4 and 1 bytes, more tiles than CTAs
EXPAND = [(1, 1, 1), (127, 63, 64), (129, 64, 65), (130, 256, 128), (300, 257, 257), (128, 1024, 256),
          (200, 1025, 300), (260, 1280, 256), (100, 1284, 70), (64, 2561, 130), (33, 4608, 65),
          (33, 4609, 65), (30000, 16, 300), (300, 1100, 449), (500, 1500, 1000), (140, 2900, 193), (2000, 700, 2100),
          (700, 300, 1500), (4000, 3000, 96), (20000, 1600, 161)]


@pytest.mark.parametrize("n,D,K", EXPAND)
@pytest.mark.parametrize("kind", ["pixels", "saturated", "sparse"])
def test_expand_edges(n, D, K, kind):
    x = W.pixel_bytes(n + D, n, D, kind)
    e = O.expand_weights(5 + K, K, D)
    E = torch.empty((K, W.words(D)), dtype=torch.int64, device=DEV)
    B.bmlp_expand_weights(5 + K, K, D, E)
    out = torch.full((n, W.words(K)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_expand_sign(torch.from_numpy(x).to(DEV), E, K, out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), W.pack(O.expand_sign(x, e)))


# a device-side wait taken as expired at a CTA's first tile, one in the middle and the
# last: the CTA's tiles are whole all the same, for each kind of copy, a short last
# tile, two neuron tiles and words past K
@pytest.mark.parametrize("tile", [0, 1, 2])
@pytest.mark.parametrize("n,D,K", [(39000, 64, 64), (20000, 132, 257), (40001, 77, 33), (70, 784, 1000)])
def test_expand_after_an_expired_wait(n, D, K, tile):
    x = W.pixel_bytes(n + D, n, D, "pixels")
    e = O.expand_weights(5 + K, K, D)
    E = torch.empty((K, W.words(D)), dtype=torch.int64, device=DEV)
    B.bmlp_expand_weights(5 + K, K, D, E)
    out = torch.full((n, W.words(K)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_debug_expand_sign(torch.from_numpy(x).to(DEV), E, K, out, tile)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), W.pack(O.expand_sign(x, e)))


# rows that start at any byte of a 32-bit word, also the first; other bytes all
# around them
@pytest.mark.parametrize("off", [0, 1, 2, 3])
@pytest.mark.parametrize("n,D,K", [(1, 1, 1), (5, 3, 70), (129, 70, 64), (300, 254, 130), (140, 255, 65), (131, 513, 257),
                                   (127, 256, 64), (50, 4607, 64)])
def test_expand_unaligned(n, D, K, off):
    x = W.pixel_bytes(n + D + off, n, D, "pixels")
    x[-1, -1] = x[0, 0] = 255
    buf = torch.full((n * D + 16,), 255, dtype=torch.uint8, device=DEV)
    buf[off:off + n * D] = torch.from_numpy(x).to(DEV).view(-1)
    e = O.expand_weights(5 + K, K, D)
    E = torch.empty((K, W.words(D)), dtype=torch.int64, device=DEV)
    B.bmlp_expand_weights(5 + K, K, D, E)
    out = torch.full((n, W.words(K)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_expand_sign(buf[off:off + n * D].view(n, D), E, K, out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), W.pack(O.expand_sign(x, e)))


# widths at every change of registers per lane and warps per pattern
@pytest.mark.parametrize("K", [1, 2, 31, 33, 256, 257, 512, 513, 800, 801, 1024, 1025, 1536, 1537, 2048, 2049, 3072, 3073,
                               4096, 4097])
@pytest.mark.parametrize("kind", ["pixels", "gauss", "ties", "wide"])
def test_binarize_edges(K, kind):
    n = 37
    if kind == "wide":   # every magnitude, infinities, constant rows, denormals
        rng = np.random.default_rng(K)
        x = (rng.standard_normal((n, K)) * 10.0 ** rng.uniform(-40, 38, (n, K))).astype(np.float32)
        x[0] = 3.0
        x[1, ::2], x[1, 1::2] = np.float32(np.inf), np.float32(-np.inf)
        x[2, : K // 2] = np.float32(-0.0)
        x[3, : K // 2 + 1], x[3, K // 2 + 1:] = np.float32(-0.0), np.float32(0.0)   # median -0
    else:
        x = W.real_patterns(K, n, K, kind)
    out = torch.full((n, W.words(K)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_binarize_median(torch.from_numpy(x).to(DEV), out)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), W.pack(O.binarize_median(x)))


# NaNs of both signs and several payloads (the padding's key among them), as few and as
# many as half: keys ordered by their bits, x > m as floats (false for a NaN)
@pytest.mark.parametrize("K", [1, 2, 33, 300, 784, 1200, 2048, 3000, 4096, 4097])
def test_binarize_nan(K):
    rng = np.random.default_rng(K)
    n = 40
    x = rng.standard_normal((n, K)).astype(np.float32)
    nans = np.array([0x7FC00000, 0xFFC00000, 0x7FFFFFFF, 0xFFFFFFFF, 0x7F800001], np.uint32).view(np.float32)
    for i in range(n):
        hit = rng.random(K) < (i % 10) / 9.0
        x[i, hit] = nans[rng.integers(0, 5, hit.sum())] if i < 20 else nans[i % 5]
    x[0, 0], x[-1] = np.inf, nans[2]
    u = x.view(np.uint32)
    key = np.where(u >> 31, ~u, u | np.uint32(1 << 31))
    m = np.sort(key, axis=1)[:, (K + 1) // 2 - 1]
    m = np.where(m >> 31, m & np.uint32(0x7FFFFFFF), ~m).astype(np.uint32).view(np.float32)
    out = torch.full((n, W.words(K)), -1, dtype=torch.int64, device=DEV)
    B.bmlp_binarize_median(torch.from_numpy(x).to(DEV), out)
    want = W.pack(np.where(x > m[:, None], 1, -1))
    assert np.array_equal(out.cpu().numpy().view(np.uint64), want)
