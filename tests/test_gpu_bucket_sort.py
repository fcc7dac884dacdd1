"""The bucket suffix sort where it can go wrong: edges of its 8192-byte
encoding tiles and 44-bit keys, buckets of every size class and above the
largest one, groups of equal keys that need one, many or too many further
keys, identical rotations. Last columns and origin rows equal the oracle's;
the flagged blocks' conditional graph nodes give the containers of the
direct call."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lfc():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


def _repeats(rng, word, sep, total):
    """word, then sep random bytes, again and again."""
    n = total // (len(word) + sep)
    out = np.empty((n, len(word) + sep), dtype=np.uint8)
    out[:, :len(word)] = np.frombuffer(word, dtype=np.uint8)
    out[:, len(word):] = rng.integers(0, 256, (n, sep), dtype=np.uint8)
    return out.tobytes()


def _inputs(name):
    rng = np.random.default_rng(99)
    if name == "tile_edges":
        return [bytes(rng.integers(0, 5, n, dtype=np.uint8)) for n in
                (1, 2, 3, 15, 16, 17, 43, 44, 45, 48, 49, 8143, 8144, 8145, 8191, 8192, 8193, 8240, 8241, 16384)]
    if name == "skewed":  # long codes next to one-bit ones
        return [bytes(np.minimum(rng.geometric(0.5, 60000), 255).astype(np.uint8)),
                bytes(np.where(rng.random(50001) < 0.001, rng.integers(0, 256, 50001), 0).astype(np.uint8))]
    if name == "identical_rotations":
        return [b"abcd" * 20, bytes(rng.integers(0, 256, 500, dtype=np.uint8)) * 20,
                bytes(rng.integers(0, 256, 1000, dtype=np.uint8)) * 33, b"ab" * 9000]
    if name == "groups":  # groups of 2, 31, 32, 33 and 60 equal keys, shared for 100 .. 3000 bytes
        out = []
        for copies, n in ((2, 3000), (31, 200), (32, 200), (33, 200), (60, 100), (5, 1500)):
            word = bytes(rng.integers(0, 256, n, dtype=np.uint8))
            out.append(b"".join(word + bytes(rng.integers(0, 256, 7, dtype=np.uint8)) for _ in range(copies)))
        return out
    # one 16-bit key prefix with about this many rotations
    n = {"class_4096": 3500, "class_8192": 6500, "class_24576": 15000, "above_classes": 30000}[name]
    return [_repeats(rng, b"qrstuvwxyz", 3, 13 * n), bytes(rng.integers(0, 256, 30000, dtype=np.uint8))]


@pytest.mark.parametrize("name", ["tile_edges", "skewed", "identical_rotations", "groups", "class_4096", "class_8192",
                                  "class_24576", "above_classes"])
def test_bwt_equals_oracle(lfc, name):
    import torch
    blocks = _inputs(name)
    plan = lfc.Plan(195, 195, 13, max_frames=24)
    data = torch.from_numpy(np.frombuffer(b"".join(blocks), dtype=np.uint8).copy()).cuda()
    sizes = [len(b) for b in blocks]
    L, ln, orig = plan.bwt_blocks(data, np.cumsum([0] + sizes)[:-1], sizes)
    L, ln, orig = L.cpu().numpy(), ln.cpu().numpy(), orig.cpu().numpy()
    for i, b in enumerate(blocks):
        r = oracle.rle1(b)
        ref, ref_row = oracle.bwt(r)
        assert int(ln[i]) == r.size
        assert np.array_equal(L[i, :r.size], ref), (name, i)
        assert int(orig[i]) == ref_row, (name, i)
    plan.close()


def test_flagged_blocks_in_a_graph(lfc):
    """Repetitive frames (every row alike; one word over and over) next to a
    noisy one: LSD passes and doubling rounds as conditional graph nodes."""
    import torch
    p, w, h = 15, 300, 300
    rng = np.random.default_rng(5)
    rows = np.tile(rng.integers(0, 4000, w).astype(np.uint16), (h, 1))
    word = np.resize(np.concatenate([np.full(9, 0x7172, np.uint16), rng.integers(0, 9, 1).astype(np.uint16)]), w * h).reshape(h, w)
    noise = rng.integers(0, 300, (h, w)).astype(np.uint16)
    frames = [np.ascontiguousarray(f) for f in (rows, noise, word)]
    plan = lfc.Plan(w, h, p, max_frames=3)
    ds = [lfc.to_device_frame(f) for f in frames]
    choice = torch.zeros(3, dtype=torch.uint8, device="cuda")
    refs = [oracle.compress_id(f, p, 0) for f in frames]
    assert plan.compress_to_bytes(ds, p, choice=choice) == refs
    batch = plan.batch(ds, p, choice=choice)
    for _ in range(2):
        batch.launch()
        torch.cuda.synchronize()
        assert batch.to_bytes() == refs
    batch.close()
    plan.close()


def _check(lfc, blocks):
    import torch
    plan = lfc.Plan(195, 195, 13, max_frames=24)
    data = torch.from_numpy(np.frombuffer(b"".join(blocks), dtype=np.uint8).copy()).cuda()
    sizes = [len(b) for b in blocks]
    L, ln, orig = plan.bwt_blocks(data, np.cumsum([0] + sizes)[:-1], sizes)
    L, ln, orig = L.cpu().numpy(), ln.cpu().numpy(), orig.cpu().numpy()
    for i, b in enumerate(blocks):
        r = oracle.rle1(b)
        ref, ref_row = oracle.bwt(r)
        assert int(ln[i]) == r.size and int(orig[i]) == ref_row, i
        assert np.array_equal(L[i, :r.size], ref), i
    plan.close()


def test_largest_class_in_a_large_pass(lfc):
    """24 blocks of at most 195 000 bytes are more than 4 M words, so the
    bucket of 15 000 words is sorted as one (a small pass takes LSD passes)."""
    rng = np.random.default_rng(7)
    _check(lfc, _inputs("class_24576") + [bytes(rng.integers(0, 30, 500 + i, dtype=np.uint8)) for i in range(22)])


@pytest.mark.parametrize("copies", [1500, 2100, 4000, 4200, 9000])
def test_group_lengths_of_the_rounds(lfc, copies):
    """Groups that stay together for several doubling rounds, around half a
    tile, a tile and the segmented sort's window: a round takes its radix
    passes only when a half tile holds no group head."""
    rng = np.random.default_rng(copies)
    word = bytes(rng.integers(97, 123, 60, dtype=np.uint8))
    _check(lfc, [_repeats(rng, word, 3, 63 * copies), bytes(rng.integers(0, 4, 20000, dtype=np.uint8))])
