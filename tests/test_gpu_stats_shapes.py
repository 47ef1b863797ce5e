"""The statistics kernels at odd sizes: frames whose rows and starts are at any alignment, every channel count, blocks
of one pixel and of the whole frame, flat frames (one large count) and coordinates outside the frame.  Counts are exact;
an entropy is a sum of at most 256 terms of a few roundings each, so it is within 1e-12 of the same sum in numpy."""
import numpy as np
import pytest
import torch

import paper_2505_07158_gb300 as fhd
from paper_2505_07158_gb300 import _lib

pytestmark = pytest.mark.gpu


def frames(count, h, w, c, flat=False, seed=5):
    g = np.random.default_rng(seed)
    a = np.full((count, h, w, c), 77, dtype=np.uint8) if flat else g.integers(0, 256, size=(count, h, w, c), dtype=np.uint8)
    return a, torch.from_numpy(a).cuda()


def entropy(x):
    z = np.bincount(x.reshape(-1), minlength=256).astype(np.float64)
    z = z[z > 0]
    return np.log2(z.sum()) - (z * np.log2(z)).sum() / z.sum()


@pytest.mark.parametrize("c", [1, 2, 3, 4])
@pytest.mark.parametrize("shape,bs", [((5, 7), 1), ((5, 7), 5), ((61, 47), 3), ((61, 47), 44), ((64, 300), 64), ((300, 300), 300)])
@pytest.mark.parametrize("flat", [False, True])
def test_local_entropy_blocks(c, shape, bs, flat):
    a, dev = frames(3, *shape, c, flat)
    g = np.random.default_rng(6)
    k = 4
    blocks = np.stack([g.integers(0, shape[0] - bs + 1, (3, k)), g.integers(0, shape[1] - bs + 1, (3, k))], -1).astype(np.int32)
    blocks[0, 0] = (shape[0] - bs, shape[1] - bs)
    out, status = _lib.fhd_stats_local_entropy(dev, torch.from_numpy(blocks).cuda(), bs)
    assert int(status) == 0
    for f in range(3):
        for ch in range(c):
            ref = np.mean([entropy(a[f, r:r + bs, q:q + bs, ch]) for r, q in blocks[f]])
            assert abs(float(out[f, ch]) - ref) < 1e-12


@pytest.mark.parametrize("block", [(-1, 0), (0, -1), (-2 ** 31, 3), (60, 0), (0, 60)])
def test_blocks_outside_are_reported(block):
    _, dev = frames(1, 61, 47, 3)
    blocks = torch.tensor([[block, (0, 0)]], dtype=torch.int32, device="cuda")
    _, status = _lib.fhd_stats_local_entropy(dev, blocks, 3)
    assert int(status) == 1


@pytest.mark.parametrize("c", [1, 2, 3, 4])
@pytest.mark.parametrize("shape,npairs", [((2, 2), 1), ((5, 7), 31), ((61, 47), 1024), ((61, 47), 1025), ((64, 300), 10000),
                                          ((300, 301), 50001)])
def test_correlation_sums(c, shape, npairs):
    a, dev = frames(3, *shape, c)
    g = np.random.default_rng(8)
    pairs = np.stack([g.integers(0, shape[0] - 1, (3, 3, npairs)), g.integers(0, shape[1] - 1, (3, 3, npairs))], -1).astype(np.int32)
    sums, r, status = _lib.fhd_stats_correlation(dev, torch.from_numpy(pairs).cuda())
    assert int(status) == 0
    for f in range(3):
        for d, (di, dj) in enumerate(((0, 1), (1, 0), (1, 1))):
            i, j = pairs[f, d, :, 0], pairs[f, d, :, 1]
            for ch in range(c):
                x, y = a[f, i, j, ch].astype(np.int64), a[f, i + di, j + dj, ch].astype(np.int64)
                assert sums[f, ch, d].tolist() == [x.sum(), y.sum(), (x * x).sum(), (y * y).sum(), (x * y).sum()]


@pytest.mark.parametrize("pair,directions", [((-1, 0), 7), ((0, -1), 7), ((60, 0), 6), ((0, 46), 5), ((61, 0), 7), ((0, 47), 7)])
def test_pairs_outside_are_reported(pair, directions):
    _, dev = frames(1, 61, 47, 3)
    for d in range(3):
        pairs = torch.zeros((1, 3, 5, 2), dtype=torch.int32)
        pairs[0, d, 2] = torch.tensor(pair, dtype=torch.int32)
        _, _, status = _lib.fhd_stats_correlation(dev, pairs.cuda())
        assert int(status) == directions >> d & 1


@pytest.mark.parametrize("c", [1, 2, 3, 4])
@pytest.mark.parametrize("count,h,w", [(1, 1, 1), (3, 1, 5), (2, 7, 13), (5, 61, 47), (2, 333, 517), (1, 1111, 1777), (40, 64, 64)])
@pytest.mark.parametrize("offset,skew", [(0, 0), (1, 0), (7, 0), (0, 3)])
def test_streaming_counts(c, count, h, w, offset, skew):
    """Every byte counted once, from any start: histograms, changed pixels and |a - b| are exact."""
    n = count * h * w * c
    g = np.random.default_rng(9)
    a, b = (g.integers(0, 256, size=n + 16, dtype=np.uint8) for _ in range(2))
    b[::3] = a[::3]
    da = torch.from_numpy(a).cuda()[offset:offset + n].view(count, h, w, c)
    db = torch.from_numpy(b).cuda()[offset + skew:offset + skew + n].view(count, h, w, c)
    a, b = a[offset:offset + n].reshape(count, h * w, c), b[offset + skew:offset + skew + n].reshape(count, h * w, c)
    hist, _ = _lib.fhd_stats_histogram(da)
    counts, _ = _lib.fhd_stats_npcr_uaci(da, db)
    hist, counts = hist.cpu().numpy(), counts.cpu().numpy()
    for f in range(count):
        for ch in range(c):
            x, y = a[f, :, ch].astype(np.int64), b[f, :, ch].astype(np.int64)
            assert np.array_equal(hist[f, ch], np.bincount(x, minlength=256))
            assert counts[f, ch].tolist() == [int((x != y).sum()), int(np.abs(x - y).sum())]
