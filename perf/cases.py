"""What a program does with this library, as cases whose time is measured: the video cipher's calls from one small
frame to a batch of 8K frames, the hot path's steps by themselves, and the frame statistics.

A case is a dict of plain values.  ``prepare`` makes what a program holds before the call (frames, keys, open
streams, output buffers), ``run`` is one pass through the public entry points, ``work`` the bytes and binary64
operations the pass cannot do without, ``exact`` the statistics in 64 bits by plain torch (the cipher's own
outputs are bytes, which are compared as they are)."""
import math

import numpy as np
import torch

import paper_2505_07158_gb300 as fhd
from paper_2505_07158_gb300._lib import fhd_frame_digest

# Frame sizes of the repository's workloads: height, width, channels.
VGA, HD, FHD, UHD, UHD8 = (480, 640, 3), (720, 1280, 3), (1080, 1920, 3), (2160, 3840, 3), (4320, 7680, 3)
MIXES = {"4k": (VGA, HD, FHD, UHD), "serving": (VGA, HD, FHD)}


def case(op, shape, frames=1, streams=1, n=32, digest="xor", transport="plain", mix="", kind="gradient"):
    """One case: `frames` frames of every one of `streams` streams, all of `shape` or of the sizes of `mix` in turn."""
    return {"op": op, "h": shape[0], "w": shape[1], "c": shape[2], "frames": frames, "streams": streams, "n": n,
            "digest": digest, "transport": transport, "mix": mix, "kind": kind}


def listed():
    named = [
        # One small frame sent and received: a thumbnail or a camera preview; launches and latency count.
        ("small_256_round_trip", case("round_trip", (256, 256, 3), kind="uniform")),
        # A grey frame of odd sides with the options that a channel may agree on (another worker count, the tree
        # digest, the masked transport): no row of it is aligned.
        ("ragged_grey_options", case("round_trip", (241, 317, 1), n=6, digest="tree", transport="masked")),
        # The plain per-frame path at the paper's size, each direction by itself: a live sender, a live receiver.
        ("frame_1080p_encrypt", case("encrypt", FHD)),
        ("frame_1080p_decrypt", case("decrypt", FHD)),
        # A second of video as one call per direction, the frames chained in one stream: a file or a recorder.
        ("clip_30x1080p_round_trip", case("round_trip", FHD, frames=30)),
        # Frames of many streams and sizes in one persistent launch of sender and receiver: a gateway.
        ("mixed_64_persistent", case("persistent", FHD, streams=64, mix="4k")),
        # One frame of every one of 32 concurrent streams in one call: what a serving step admits.
        ("serving_32_streams_encrypt", case("encrypt", FHD, streams=32, mix="serving")),
        # Large frames, half of them noise, sent and received: the stress load.
        ("stress_8k_round_trip", case("round_trip", UHD8, frames=4, kind="halves")),
        # The integrity digests of a batch of frames by themselves: an archive that is checked.
        ("digest_16x720p", case("digest", HD, frames=16)),
        # The confusion and XOR both ways by themselves, distances and bytes given: a program with a keystream.
        ("permute_4k_both_ways", case("permute", UHD, kind="uniform")),
        # The worker pairs from any iterates, as the paper's Algorithm 2 states them.
        ("worker_pairs_720p", case("pairs", HD)),
        # The evaluation's statistics of a clip and of its ciphertext-like noise: histogram, NPCR and UACI,
        # correlation of 10,000 pairs a direction, local entropy of 30 blocks of 44 x 44.
        ("statistics_30x1080p", case("statistics", FHD, frames=30, kind="uniform")),
    ]
    return [dict(c, name=name) for name, c in named]


def draw(rng):
    """One more case: a call of the listed ones at a size spread over the logarithm of its range, odd sides
    among them, no dearer than the largest listed."""
    def side(lo, hi):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return v if rng.random() < 0.5 else max(16, v - v % 16)

    op = rng.choice(("round_trip", "round_trip", "encrypt", "decrypt", "persistent", "digest", "permute", "pairs",
                     "statistics"))
    c = rng.choice((3, 3, 3, 1, 4))
    if op == "pairs":
        shape = (side(64, 720), side(64, 1280), c)
    elif op == "statistics":
        shape = (side(64, 2160), side(64, 3840), c)
    else:
        shape = (side(64, 2160), side(64, 3840), c)
    most = max(1, min(64, int(1.5e8 / (shape[0] * shape[1] * shape[2]))))
    count = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most)))))) if most > 1 else 1
    if op in ("permute", "pairs"):
        count = 1
    streams = count if op == "persistent" or (op in ("encrypt", "round_trip") and rng.random() < 0.4) else 1
    plain = op in ("digest", "permute", "pairs", "statistics")
    n = 32 if op in ("permute", "statistics") else rng.choice((32, 32, 32, 8, 64, 100))
    return case(op, shape, frames=count // streams, streams=streams, n=n,
                digest="xor" if plain and op != "digest" else rng.choice(("xor", "xor", "tree")),
                transport="plain" if plain else rng.choice(("plain", "plain", "masked")),
                kind=rng.choice(("gradient", "uniform")))


# ---- inputs

def shapes_of(case):
    """The frames' shapes in call order: stream by stream, `frames` of each."""
    mix = MIXES.get(case["mix"], ((case["h"], case["w"], case["c"]),))
    return [mix[s % len(mix)] for s in range(case["streams"]) for _ in range(case["frames"])]


def frame(shape, t, kind, g):
    """One uint8 frame on the GPU: uniform bytes, or a smooth gradient that moves 2 pixels a frame with noise of
    standard deviation 8."""
    h, w, c = shape
    if kind == "uniform":
        return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=g)
    a = (torch.arange(c, device="cuda") + 1) / (c + 1)
    i = torch.arange(h, device="cuda", dtype=torch.float32)[:, None, None] / h
    j = torch.remainder(torch.arange(w, device="cuda", dtype=torch.float32) + 2 * t, w)[None, :, None] / w
    x = torch.randn(shape, device="cuda", generator=g).mul_(8.0)
    x += 255.0 * (a * i + (1 - a) * j)
    return x.round_().clamp_(0, 255).to(torch.uint8)


def frames_of(case, g):
    shapes = shapes_of(case)
    kinds = [case["kind"]] * len(shapes)
    if case["kind"] == "halves":
        kinds = ["uniform" if k < len(shapes) // 2 else "gradient" for k in range(len(shapes))]
    return [frame(s, k % case["frames"], kinds[k], g) for k, s in enumerate(shapes)]


class Buffers:
    """One flat output buffer with a view per frame, each on a 256-byte boundary, as a frame pool lays them out."""

    def __init__(self, shapes):
        sizes = [int(np.prod(s)) for s in shapes]
        at = np.concatenate([[0], np.cumsum([(b + 255) // 256 * 256 for b in sizes])]).tolist()
        self.flat = torch.zeros(at[-1], dtype=torch.uint8, device="cuda")
        self.views = [self.flat[o:o + b].view(s) for o, b, s in zip(at, sizes, shapes)]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    op, shapes = case["op"], shapes_of(case)
    h, w, c = shapes[0]
    st = {"case": dict(case)}
    if op == "digest":
        st["data"] = torch.stack(frames_of(case, g))
        return st
    if op == "permute":
        st["F"] = frames_of(case, g)[0]
        st["D"] = torch.randint(-32768, 32768, (c * (h + w),), dtype=torch.int16, device="cuda", generator=g)
        st["B"] = torch.randint(0, 256, (h * w * c,), dtype=torch.uint8, device="cuda", generator=g)
        return st
    if op == "pairs":
        u = torch.tensor([20.0, 20.0, 40.0, 20.0], dtype=torch.float64, device="cuda")
        st["IR"] = torch.rand((2 * case["n"], 4), dtype=torch.float64, device="cuda", generator=g) * u
        st["gamma"] = float(rng.uniform(-1.52, -0.06))
        return st
    if op == "statistics":
        n = case["frames"]
        st["a"] = torch.stack(frames_of(case, g))
        st["b"] = torch.randint(0, 256, (n, h, w, c), dtype=torch.uint8, device="cuda", generator=g)
        st["pairs"] = torch.stack([torch.randint(0, h - 1, (n, 3, 10000), device="cuda", generator=g),
                                   torch.randint(0, w - 1, (n, 3, 10000), device="cuda", generator=g)], dim=-1).int()
        st["blocks"] = torch.stack([torch.randint(0, h - 43, (n, 30), device="cuda", generator=g),
                                    torch.randint(0, w - 43, (n, 30), device="cuda", generator=g)], dim=-1).int()
        return st
    # the cipher's calls: a sender and a receiver, a stream (with its own key) for every video
    key = rng.integers(0, 256, size=32, dtype=np.uint8).tobytes()
    opts = dict(n_workers=case["n"], digest_mode=case["digest"], digest_transport=case["transport"])
    enc, dec = fhd.Cipher(key, **opts), fhd.Cipher(key, **opts)
    keys = [rng.integers(0, 256, size=32, dtype=np.uint8).tobytes() for _ in range(case["streams"])]
    sids, rids = [enc.open_stream(k) for k in keys], [dec.open_stream(k) for k in keys]
    F, E, P = frames_of(case, g), Buffers(shapes), Buffers(shapes)
    H = torch.zeros((len(shapes), 32), dtype=torch.uint8, device="cuda")
    of = [k // case["frames"] for k in range(len(shapes))]
    st.update(enc=enc, dec=dec, E=E, P=P, H=H, F=F,
              send=[(sids[of[k]], F[k], E.views[k], H[k]) for k in range(len(shapes))],
              receive=[(rids[of[k]], E.views[k], P.views[k], H[k]) for k in range(len(shapes))])
    if op == "decrypt":   # what a receiver is handed: ciphertext and digest
        enc.encrypt_frames(st["send"])
        if case["transport"] == "masked":   # a receiver unmasks the digest in place: each pass gets it as sent
            st["sent"] = H.clone()
    return st


# ---- one pass.  Every pass of the cipher's calls continues its streams, as the next frames of a video would (a
# receiver that is handed the same ciphertext again decrypts it with the next state, at the same cost).

def run(state):
    case, op = state["case"], state["case"]["op"]
    if op == "digest":
        return fhd_frame_digest(state["data"], n=case["n"], count=case["frames"], mode=case["digest"])
    if op == "permute":
        E = fhd.fhd_permute_encrypt(state["F"], state["D"], state["B"])
        return {"E": E, "P": fhd.fhd_permute_decrypt(E, state["D"], state["B"])}
    if op == "pairs":
        D, B = fhd.fhd_keystream(state["IR"], state["gamma"], case["h"], case["w"], case["c"], n_workers=case["n"])
        return {"D": D, "B": B}
    if op == "statistics":
        hist, st = fhd.fhd_stats_histogram(state["a"])
        counts, np_ua = fhd.fhd_stats_npcr_uaci(state["a"], state["b"])
        sums, r, bad = fhd.fhd_stats_correlation(state["a"], state["pairs"])
        ent, bad2 = fhd.fhd_stats_local_entropy(state["a"], state["blocks"], 44)
        return {"hist": hist, "stats": st, "counts": counts, "npcr_uaci": np_ua, "sums": sums, "r": r, "bad": bad,
                "entropy": ent, "bad2": bad2}
    if op == "persistent":
        state["enc"].round_trip_persistent(state["dec"], state["send"], state["receive"])
    if op in ("encrypt", "round_trip"):
        state["enc"].encrypt_frames(state["send"])
    if op == "decrypt" and "sent" in state:
        state["H"].copy_(state["sent"])
    if op in ("decrypt", "round_trip"):
        state["dec"].decrypt_frames(state["receive"])
    out = {"H": state["H"]}
    if op != "decrypt":
        out["E"] = state["E"].flat
    if op != "encrypt":
        out["P"] = state["P"].flat
    return out


# ---- what a pass cannot do without

def chain_ops(shape, n):
    """Binary64 operations of the distinct states a frame's keystream is made of: 2n of LHCS_m and those that the
    longest worker slice takes, 104 operations each."""
    h, w, c = shape
    need = 2 * -(-(c * (h + w)) // n) + -(-(h * w * c) // n)
    return 104.0 * (2 * n + -(-need // 24))


def work(case):
    op, shapes = case["op"], shapes_of(case)
    nbytes = float(sum(h * w * c for h, w, c in shapes))
    h, w, c = shapes[0]
    if op == "digest":
        return {"bytes": nbytes + 32.0 * len(shapes), "flops": 0.0}
    if op == "permute":
        return {"bytes": 2 * (3 * nbytes + 2.0 * c * (h + w)), "flops": 0.0}
    if op == "pairs":
        steps = -(-(2 * -(-(c * (h + w)) // case["n"]) + -(-(h * w * c) // case["n"])) // 24)
        return {"bytes": nbytes + 2.0 * c * (h + w) + 64.0 * case["n"], "flops": 104.0 * 2 * case["n"] * steps}
    if op == "statistics":
        sampled = len(shapes) * (3 * 10000 * (8 + 2.0 * c) + 30 * (8 + 44 * 44 * c))
        return {"bytes": 2 * nbytes + sampled + len(shapes) * c * 256 * 4.0, "flops": 0.0}
    ways = 2 if op in ("round_trip", "persistent") else 1
    return {"bytes": ways * (2 * nbytes + 32.0 * len(shapes)),
            "flops": ways * sum(chain_ops(s, case["n"]) for s in shapes)}


# ---- the computed numbers in 64 bits, by plain torch

def exact(case, seed):
    if case["op"] != "statistics":
        return None
    st = prepare(case, seed)
    a, b = st["a"], st["b"]
    n, h, w, c = a.shape
    stats, np_ua = torch.zeros((n, c, 3), dtype=torch.float64), torch.zeros((n, c, 2), dtype=torch.float64)
    r, ent = torch.zeros((n, c, 3), dtype=torch.float64), torch.zeros((n, c), dtype=torch.float64)
    for f in range(n):
        for k in range(c):
            x, y = a[f, :, :, k].reshape(-1).long(), b[f, :, :, k].reshape(-1).long()
            z = torch.bincount(x, minlength=256).double()
            p = z / z.sum()
            stats[f, k, 0] = ((z - z.mean()) ** 2).mean()
            stats[f, k, 1] = ((z - z.mean()) ** 2 / z.mean()).sum()
            stats[f, k, 2] = -(p[p > 0] * torch.log2(p[p > 0])).sum()
            np_ua[f, k, 0] = 100.0 * (x != y).double().mean()
            np_ua[f, k, 1] = 100.0 * (x - y).abs().double().mean() / 255.0
            for d, (di, dj) in enumerate(((0, 1), (1, 0), (1, 1))):
                i, j = st["pairs"][f, d, :, 0].long(), st["pairs"][f, d, :, 1].long()
                u, v = a[f, i, j, k].double(), a[f, i + di, j + dj, k].double()
                u, v = u - u.mean(), v - v.mean()
                r[f, k, d] = (u * v).sum() / torch.sqrt((u * u).sum() * (v * v).sum())
            es = []
            for q in range(st["blocks"].shape[1]):
                i, j = (int(t) for t in st["blocks"][f, q])
                z = torch.bincount(a[f, i:i + 44, j:j + 44, k].reshape(-1).long(), minlength=256).double()
                p = z[z > 0] / z.sum()
                es.append(-(p * torch.log2(p)).sum())
            ent[f, k] = torch.stack(es).mean()
    return {"hist": None, "stats": stats, "counts": None, "npcr_uaci": np_ua, "sums": None, "r": r, "bad": None,
            "entropy": ent, "bad2": None}
