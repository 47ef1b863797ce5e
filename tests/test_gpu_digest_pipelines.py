"""Digest pipelines: messages at every alignment and of every length round a block and a 16-byte piece, and launches
on both sides of the line between split and unsplit messages, against hashlib (bytes are equal or wrong)."""
import hashlib

import pytest
import torch

import paper_2505_07158_gb300 as fhd
from paper_2505_07158_gb300._lib import fhd_frame_digest

pytestmark = pytest.mark.gpu

LENGTHS = sorted({max(1, e + d) for e in (16, 32, 56, 64, 80, 96, 128, 144, 192, 256, 320, 448, 1024) for d in (-1, 0, 1, 8, 15)})


def reference(buf: bytes, n: int) -> bytes:
    acc = 0
    for i in range(n):
        h = hashlib.sha256(buf[i * len(buf) // n:(i + 1) * len(buf) // n]).digest()
        acc ^= int.from_bytes(h, "big")
    return acc.to_bytes(32, "big")


@pytest.fixture(scope="module")
def data():
    g = torch.Generator().manual_seed(41)
    host = torch.randint(0, 256, (1 << 21,), dtype=torch.uint8, generator=g)
    return host, host.cuda()


@pytest.mark.parametrize("offset", range(16))
def test_alignment_and_length(data, offset):
    host, dev = data
    for length in LENGTHS:
        got = bytes(fhd_frame_digest(dev[offset:offset + length], n=1)[0].cpu().numpy())
        assert got == hashlib.sha256(host[offset:offset + length].numpy().tobytes()).digest(), (offset, length)


@pytest.mark.parametrize("n,length,offset", [(2, 3, 0), (5, 4, 1), (6, 12733 * 6 - 1, 0), (31, 31 * 90 + 7, 3), (32, 100001, 0),
                                             (33, 33 * 64, 0), (33, 33 * 67 + 5, 9), (1024, 1024 * 70 + 513, 2)])
def test_mixed_messages_of_a_pipeline(data, n, length, offset):
    host, dev = data
    got = bytes(fhd_frame_digest(dev[offset:offset + length], n=n)[0].cpu().numpy())
    assert got == reference(host[offset:offset + length].numpy().tobytes(), n)


@pytest.mark.parametrize("count,n", [(152, 32), (153, 32), (303, 16), (305, 16), (1024, 6), (4864, 1), (4865, 1)])
@pytest.mark.parametrize("nbytes", [208, 333])
def test_both_sides_of_the_split(data, count, n, nbytes):
    host, dev = data
    got = fhd_frame_digest(dev[:count * nbytes], n=n, count=count).cpu()
    raw = host.numpy()
    for k in range(0, count, 7):
        assert bytes(got[k].numpy()) == reference(raw[k * nbytes:(k + 1) * nbytes].tobytes(), n), k
