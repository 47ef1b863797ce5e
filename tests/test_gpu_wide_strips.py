"""The column pass where a strip row has more bytes than the CTA has threads (a wide strip of a frame that takes the
bytewise route, 256 threads): set by hand, at a batch's built-in width, and in a batch whose largest frame brings the
256 threads.  Against the oracle; bytes are equal or wrong."""
import numpy as np
import pytest
import torch

import oracle
import paper_2505_07158_gb300 as fhd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,P", [((241, 317, 3), 128), ((241, 317, 3), 86), ((61, 131, 4), 128), ((61, 131, 3), 85)])
def test_a_width_set_by_hand(shape, P):
    """QC = 384, 258 (two bytes beyond the threads), 512 and, in the last strip of 131 columns, a remainder."""
    g = np.random.default_rng(P)
    h, w, c = shape
    F, B = (g.integers(0, 256, size=shape, dtype=np.uint8) for _ in range(2))
    D = g.integers(0, 65536, size=c * (h + w), dtype=np.uint16)
    dev = [torch.from_numpy(x).cuda() for x in (F, D.view(np.int16), B)]
    fhd.fhd_set_strip_width(*shape, P)
    fhd.fhd_set_cta_threads(*shape, 256, 0)
    try:
        E = fhd.fhd_permute_encrypt(*dev)
        assert np.array_equal(E.cpu().numpy(), oracle.permute_encrypt(F, D, B))
        assert np.array_equal(fhd.fhd_permute_decrypt(E, *dev[1:]).cpu().numpy(), F)
    finally:
        fhd.fhd_set_strip_width(*shape, 0)
        fhd.fhd_set_cta_threads(*shape, 0, 0)


@pytest.mark.parametrize("shapes,largest", [([(241, 317, 3)] * 30, (241, 317, 3)),
                                            ([(241, 317, 3)] * 30 + [(480, 640, 3)], (480, 640, 3))])
def test_batches_at_the_built_in_width(shapes, largest):
    """Enough strips that no frame's are narrowed: 128 columns of 3 bytes, with the 256 threads of the largest frame."""
    g = np.random.default_rng(len(shapes))
    key = bytes(range(32))
    fhd.fhd_set_cta_threads(*largest, 256, 0)
    try:
        enc, dec = fhd.Cipher(key, n_workers=256), fhd.Cipher(key, n_workers=256)
        sid, rid = enc.open_stream(), dec.open_stream()
        F = [torch.from_numpy(g.integers(0, 256, size=s, dtype=np.uint8)).cuda() for s in shapes]
        E, P = [torch.zeros_like(f) for f in F], [torch.zeros_like(f) for f in F]
        H = torch.zeros((len(F), 32), dtype=torch.uint8, device="cuda")
        enc.encrypt_frames([(sid, f, e, h) for f, e, h in zip(F, E, H)])
        ref = oracle.Stream.from_key(key, n=256)
        for f, e, h in zip(F, E, H):
            E_ref, H_ref = ref.encrypt(f.cpu().numpy())
            assert bytes(h.cpu().numpy()) == H_ref and np.array_equal(e.cpu().numpy(), E_ref)
        dec.decrypt_frames([(rid, e, p, h) for e, p, h in zip(E, P, H)])
        assert all(torch.equal(p, f) for p, f in zip(P, F))
    finally:
        fhd.fhd_set_cta_threads(*largest, 0, 0)
