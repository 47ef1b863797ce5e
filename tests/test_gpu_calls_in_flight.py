"""What calls cost beside other calls, and on inputs that a fast path does not suit: ratios of times within one process
(the fastest of several passes), each with a bar between what the call takes and what it took where it went wrong."""
import hashlib
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
import paper_2505_07158_gb300 as fhd
from paper_2505_07158_gb300 import _lib

pytestmark = pytest.mark.gpu
# the checked build's kernels take other times
timed = pytest.mark.skipif(fhd.checked_requested(), reason="times of the default build")


def fastest(fn, reps=6):
    """Milliseconds of the fastest pass of fn, the first two not counted."""
    out = []
    for _ in range(reps + 2):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b))
    return min(out[2:])


def on_streams(streams, call):
    """call(i, stream) on every stream, forked from and joined to the current one."""
    start = torch.cuda.Event()
    start.record()
    for i, s in enumerate(streams):
        s.wait_event(start)
        call(i, s)
    for s in streams:
        torch.cuda.current_stream().wait_stream(s)


def noise(*shape, seed=1):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=g)


@timed
def test_calls_on_more_streams_than_hardware_queues():
    """Twelve encryption calls of 8 frames on twelve streams (8 hardware queues by default): two rounds of the queues at
    most (1.9 times one round of 8 calls; 3.1 where a kernel held its queue)."""
    made = []
    for k in range(12):
        c = fhd.Cipher(bytes(range(32)))
        c.set_partition(False)
        F = noise(8, 720, 1280, 3, seed=k)
        E, H = torch.empty_like(F), torch.zeros((8, 32), dtype=torch.uint8, device="cuda")
        made.append((c, [(c.open_stream(), F[i], E[i], H[i]) for i in range(8)]))
    S = [torch.cuda.Stream() for _ in made]
    t = [fastest(lambda: on_streams(S[:n], lambda i, s: made[i][0].encrypt_frames(made[i][1], stream=s))) for n in (8, 12)]
    for c, _ in made:
        c.close()
    assert t[1] < 2.4 * t[0], t


def digests(X, streams):
    out = [torch.zeros((x.shape[0], 32), dtype=torch.uint8, device="cuda") for x in X]
    on_streams(streams, lambda i, s: fhd.fhd_frame_digest(X[i], n=32, count=X[i].shape[0], out=out[i], stream=s))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("nbytes", [1 << 20, 1000003])
def test_digests_of_pipelines_that_come_to_share_an_sm(nbytes):
    """Digests of 12 streams in flight, 360 pipelines on 152 SMs: the first ones start with two lanes per message and go
    on with one when the others arrive, at blocks that the arrival decides.  Against hashlib."""
    X = [noise(30, nbytes, seed=k) for k in range(12)]
    for x, d in zip(X, digests(X, [torch.cuda.Stream() for _ in X])):
        for buf, got in zip(x.cpu().numpy(), d.cpu().numpy()):
            acc = 0
            for i in range(64):
                lo, hi = nbytes * i // 32, nbytes * (i + 1) // 32
                acc ^= int.from_bytes(hashlib.sha256(buf[lo:hi].tobytes()).digest(), "big")
            assert got.tobytes() == acc.to_bytes(32, "big")


@timed
def test_digest_time_of_pipelines_that_share_an_sm():
    """240 pipelines of two calls on 152 SMs against the 120 of one call, two lanes per message (1.2 times; 1.55
    where every pipeline keeps two lanes per message)."""
    X = [noise(120, 720 * 1280 * 3, seed=k) for k in range(2)]
    S = [torch.cuda.Stream() for _ in X]
    t = [fastest(lambda: digests(X[:n], S[:n])) for n in (1, 2)]
    assert t[1] < 1.45 * t[0], t


def pairs_of(count, h, w, npairs):
    g = torch.Generator(device="cuda").manual_seed(npairs)
    return torch.stack([torch.randint(0, h - 1, (count, 3, npairs), device="cuda", generator=g),
                        torch.randint(0, w - 1, (count, 3, npairs), device="cuda", generator=g)], dim=-1).int()


@timed
def test_correlation_time_of_many_frames():
    """1,025 pairs of each of 1,000 frames against 1,024: the pairs of a direction are not spread over more CTAs where the
    frames fill the GPU by themselves (equal; 5 times where they were)."""
    a = noise(1000, 32, 32, 3)
    pairs = [pairs_of(1000, 32, 32, n) for n in (1024, 1025)]
    t = [fastest(lambda: [_lib.fhd_stats_correlation(a, p) for _ in range(10)]) for p in pairs]
    assert t[1] < 1.5 * t[0], t


@pytest.mark.parametrize("count,npairs", [(1, 1025), (1, 2049), (1, 4097), (30, 10000), (51, 7000), (100, 2048), (180, 7000)])
def test_correlation_sums_by_any_number_of_ctas(count, npairs):
    """Two, four and eight CTAs to a frame's direction, and one: exact sums."""
    h, w = 37, 53
    a, p = noise(count, h, w, 3, seed=count), pairs_of(count, h, w, npairs)
    sums, _, status = _lib.fhd_stats_correlation(a, p)
    assert int(status) == 0
    f = torch.arange(count, device="cuda")[:, None]
    for d, (di, dj) in enumerate(((0, 1), (1, 0), (1, 1))):
        i, j = p[:, d, :, 0].long(), p[:, d, :, 1].long()
        x, y = a[f, i, j].long(), a[f, i + di, j + dj].long()
        ref = torch.stack([x.sum(1), y.sum(1), (x * x).sum(1), (y * y).sum(1), (x * y).sum(1)], dim=-1)
        assert torch.equal(sums[:, :, d], ref)


@timed
def test_local_entropy_time_of_flat_blocks():
    """100 blocks of 16 x 16 of each of 300 flat frames against noise frames: a flat block has one logarithm to take, a
    noise block a dozen (no dearer; 1.75 times where every count up to the largest
    had its logarithm)."""
    g = torch.Generator(device="cuda").manual_seed(3)
    blocks = torch.randint(0, 49, (300, 100, 2), device="cuda", generator=g).int()
    rough = noise(300, 64, 64, 3)
    t = [fastest(lambda: _lib.fhd_stats_local_entropy(a, blocks, 16)) for a in (rough, torch.zeros_like(rough))]
    assert t[1] < 1.4 * t[0], t


@timed
def test_chain_time_at_gammas_beyond_the_attractors():
    """2,048 steps of LHCS_m at a gamma whose states leave the integer step's ranges, against one that it does not take
    at all, binary64 throughout (equal; 1.8 times where every step was tried on the integer pipes first)."""
    H = noise(32)
    t = []
    for gamma in (-1.0, 0.9):
        st = torch.tensor([12.3, 4.5, 23.4, 7.8, gamma], dtype=torch.float64, device="cuda")
        t.append(fastest(lambda: fhd.fhd_master(st, H, n_workers=1024)))
    assert t[1] < 1.25 * t[0], t


@timed
def test_worker_pair_time_of_short_slices():
    """304 pairs of 21 steps each from iterates off the attractor against 305 x 2, which the binary64 kernel takes: as
    long (1.06 times; 1.28 where the short slices took the integer step)."""
    g = torch.Generator(device="cuda").manual_seed(2)
    scale = torch.tensor([20.0, 20.0, 40.0, 20.0], dtype=torch.float64, device="cuda")
    t = []
    for n in (610, 304):
        IR = torch.rand((2 * n, 4), dtype=torch.float64, device="cuda", generator=g) * scale
        t.append(fastest(lambda: [fhd.fhd_keystream(IR, -0.9123, n, 500, 1, n_workers=n) for _ in range(30)]))
    assert t[1] < 1.15 * t[0], t


@pytest.mark.parametrize("n,w", [(1, 23), (8, 23), (9, 23), (9, 1140), (9, 1150), (32, 1100), (32, 1200), (304, 1150), (608, 1150)])
def test_worker_pairs_on_both_sides_of_the_short_slices(n, w):
    """Few pairs and many, slices of one step and on both sides of 48, against the oracle."""
    g = np.random.default_rng(n + w)
    IR = g.uniform(0, 1, (2 * n, 4)) * [20, 20, 40, 20]
    D_ref, B_ref = oracle.keystream(IR, -0.9123, n, w, 1, n, 0.01)
    D, B = fhd.fhd_keystream(torch.from_numpy(IR).cuda(), -0.9123, n, w, 1, n_workers=n)
    assert np.array_equal(D.cpu().numpy().view(np.uint16), D_ref)
    assert np.array_equal(B.cpu().numpy().reshape(-1), np.asarray(B_ref).reshape(-1))


@timed
def test_chain_time_on_the_attractor():
    """The integer step is what runs, and few of its steps are done again: 2,048 steps at gamma = -0.9123 against -1, which
    it does not take (0.68 times)."""
    H = noise(32)
    t = []
    for gamma in (-1.0, -0.9123):
        st = torch.tensor([12.3, 4.5, 23.4, 7.8, gamma], dtype=torch.float64, device="cuda")
        t.append(fastest(lambda: fhd.fhd_master(st, H, n_workers=1024)))
    assert t[1] < 0.8 * t[0], t


MANY_STREAMS = """
import time, torch
import paper_2505_07158_gb300 as fhd
h, w, c = 1081, 1917, 3
g = torch.Generator(device="cuda").manual_seed(1)
F = [torch.randint(0, 256, (h, w, c), dtype=torch.uint8, device="cuda", generator=g) for _ in range(32)]
D = torch.randint(-32768, 32768, (c * (h + w),), dtype=torch.int16, device="cuda", generator=g)
O, B, S = [torch.empty_like(f) for f in F], F[0].clone(), [torch.cuda.Stream() for _ in F]
t = []
for n in (1, 32):
    passes = []
    for _ in range(12):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for i in range(64):
            fhd.fhd_permute_decrypt(F[i % 32], D, B, out=O[i % 32], stream=S[i % n])
        torch.cuda.synchronize()
        passes.append(time.perf_counter() - t0)
    t.append(min(passes[2:]))
print("times", *t)
"""


@timed
def test_decrypting_passes_on_many_streams():
    """64 decrypting passes on 32 streams with hardware queues of their own against the same 64 on one stream: half the
    time (1.8 times it where the temporary frames came from CUDA's default pool, whose search for other streams' freed
    blocks held the caller up)."""
    env = dict(os.environ, CUDA_DEVICE_MAX_CONNECTIONS="32")
    r = subprocess.run([sys.executable, "-c", MANY_STREAMS], env=env, capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr
    t = [float(x) for x in r.stdout.split("times")[1].split()]
    assert t[1] < 1.1 * t[0], t


UNDER_CAPTURE = """
import sys, threading, torch
import paper_2505_07158_gb300 as fhd
h, w, c = 61, 67, 3
g = torch.Generator(device="cuda").manual_seed(1)
F, B = (torch.randint(0, 256, (h, w, c), dtype=torch.uint8, device="cuda", generator=g) for _ in range(2))
D = torch.randint(-32768, 32768, (c * (h + w),), dtype=torch.int16, device="cuda", generator=g)
E, P, E2, P2 = (torch.zeros_like(F) for _ in range(4))
s2 = torch.cuda.Stream()

def both(e, p, s):
    fhd.fhd_permute_encrypt(F, D, B, out=e, stream=s)
    fhd.fhd_permute_decrypt(e, D, B, out=p, stream=s)

x = torch.zeros(4, device="cuda")
x += 1
torch.cuda.synchronize()
G = torch.cuda.CUDAGraph()
with torch.cuda.graph(G, capture_error_mode="thread_local"):
    if sys.argv[1] == "captured":
        both(E, P, torch.cuda.current_stream())
    else:   # another thread's first calls while this one captures
        t = threading.Thread(target=both, args=(E2, P2, s2))
        t.start()
        t.join()
        x += 1
if sys.argv[1] == "captured":
    for _ in range(2):
        E.zero_(), P.zero_()
        G.replay()
        torch.cuda.synchronize()
        assert torch.equal(P, F)
else:
    torch.cuda.synchronize()
    assert torch.equal(P2, F)
both(E2, P2, s2)
torch.cuda.synchronize()
assert torch.equal(P2, F) and (sys.argv[1] != "captured" or torch.equal(E2, E))
"""


@pytest.mark.parametrize("who", ["captured", "beside"])
def test_permutation_under_capture(who):
    """A process's first calls captured into a graph, and its first calls beside another thread's capture."""
    r = subprocess.run([sys.executable, "-c", UNDER_CAPTURE, who], capture_output=True, text=True, timeout=300,
                       cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert r.returncode == 0, r.stderr
