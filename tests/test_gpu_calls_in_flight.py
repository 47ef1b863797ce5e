"""What calls cost beside other calls, and on inputs that a fast path does not suit: ratios of times within one process
(the fastest of several passes), each with at least a quarter between the bar and what either side of it measures."""
import pytest
import torch

import paper_2505_07158_gb300 as fhd

pytestmark = pytest.mark.gpu


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
