"""The column pass at every strip width and CTA shape, and the widths that a launch takes by itself, against the oracle
(bytes are equal or wrong): heights and strips at the edges of the column-word layout, rotations that wrap."""
import numpy as np
import pytest
import torch

import oracle
import paper_2505_07158_gb300 as fhd

pytestmark = pytest.mark.gpu

SHAPES = [(4, 16, 3), (8, 7, 4), (12, 33, 1), (20, 24, 2), (64, 100, 1), (241, 317, 1), (244, 316, 3), (240, 320, 4), (1028, 64, 3),
          (4320, 48, 3), (720, 1280, 3), (1081, 131, 3)]


def inputs(shape, seed=3):
    g = np.random.default_rng(seed)
    h, w, c = shape
    F, B = (g.integers(0, 256, size=shape, dtype=np.uint8) for _ in range(2))
    return F, g.integers(0, 65536, size=c * (h + w), dtype=np.uint16), B


def check(shape):
    F, D, B = inputs(shape)
    dev = [torch.from_numpy(x.view(np.int16) if x.dtype == np.uint16 else x).cuda() for x in (F, D, B)]
    dev[1] = dev[1].view(torch.uint16)
    E = fhd.fhd_permute_encrypt(*dev)
    assert np.array_equal(E.cpu().numpy(), oracle.permute_encrypt(F, D, B))
    assert np.array_equal(fhd.fhd_permute_decrypt(E, *dev[1:]).cpu().numpy(), F)


@pytest.mark.parametrize("shape", SHAPES)
def test_width_of_a_lone_frame(shape):
    check(shape)


@pytest.mark.parametrize("threads", [256, 512])
@pytest.mark.parametrize("P", [2, 4, 8, 12, 16, 20, 32, 64, 128])
@pytest.mark.parametrize("shape", SHAPES)
def test_every_width(shape, P, threads):
    fhd.fhd_set_strip_width(*shape, P)   # a width that does not fit is passed over
    fhd.fhd_set_cta_threads(*shape, threads, 0)
    try:
        check(shape)
    finally:
        fhd.fhd_set_strip_width(*shape, 0)
        fhd.fhd_set_cta_threads(*shape, 0, 0)


@pytest.mark.parametrize("shape", [(60, 68, 4), (61, 67, 4), (64, 256, 4), (64, 256, 3), (33, 300, 1), (1028, 128, 4)])
def test_strips_of_a_persistent_launch(shape):
    """The widest strips for the permutation group's threads, word and byte routes, against the plain path."""
    g = np.random.default_rng(7)
    key = g.integers(0, 256, size=32, dtype=np.uint8).tobytes()
    F = torch.from_numpy(g.integers(0, 256, size=shape, dtype=np.uint8)).cuda()
    out = []
    for persistent in (False, True):
        c = fhd.Cipher(key)
        s, E, H = c.open_stream(key), torch.empty_like(F), torch.zeros(32, dtype=torch.uint8, device="cuda")
        (c.encrypt_frames_persistent if persistent else c.encrypt_frames)([(s, F, E, H)])
        d = fhd.Cipher(key)
        P = torch.empty_like(F)
        (d.decrypt_frames_persistent if persistent else d.decrypt_frames)([(d.open_stream(key), E, P, H)])
        assert torch.equal(P, F)
        out.append(E)
    assert torch.equal(out[0], out[1])
