"""Blocks that repeat a shorter string, or nearly do: the origin row among
identical rotations, decoding blocks whose rows form several cycles, the
pieces of the inverse BWT where a row keeps its place among 48 k or 64 k rows, and the
suffix sort's time on long repeats."""
import bz2

import numpy as np
import pytest

import oracle


def _rows(m, L):
    """Rows in the order of a stable sort of L: where every row leads."""
    nxt = np.empty(m, dtype=np.int64)
    nxt[np.argsort(L, kind="stable")] = np.arange(m)
    return nxt


@pytest.fixture(scope="module")
def lfc():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


def _bwt_equals_oracle(lfc, blocks):
    import torch
    plan = lfc.Plan(195, 195, 13, max_frames=24)
    for a in range(0, len(blocks), plan.block_capacity):
        part = blocks[a:a + plan.block_capacity]
        data = torch.from_numpy(np.frombuffer(b"".join(part), dtype=np.uint8).copy()).cuda()
        sizes = [len(b) for b in part]
        L, ln, orig = plan.bwt_blocks(data, np.cumsum([0] + sizes)[:-1], sizes)
        L, ln, orig = L.cpu().numpy(), ln.cpu().numpy(), orig.cpu().numpy()
        for i, b in enumerate(part):
            r = oracle.rle1(b)
            ref, ref_row = oracle.bwt(r)
            assert int(ln[i]) == r.size
            assert np.array_equal(L[i, :r.size], ref), b
            assert int(orig[i]) == ref_row, b
    plan.close()


# Words with long runs of a short unit: some of the repeated block's rotations
# share a key with more than 32 others (prefix doubling orders them), some
# with their identical ones alone (further keys do).
_WORDS = [(b"a\0" * 6 + b"ad\0a\0aff" + b"\0a" * 17 + b"\0", 12),
          (b"ba" * 10 + b"bdd" + b"ab" * 30 + b"ff" + b"ab" * 20 + b"a", 4),
          (b"bca" * 5 + b"bcf" + b"abc" * 6 + b"a", 12),
          (b"\0\0a" * 11 + b"dd" + b"\0\0a" * 13 + b"dd", 8)]


@pytest.mark.gpu
def test_origin_row_of_repeated_words(lfc):
    rng = np.random.default_rng(61)
    blocks = [w * r for w, r in _WORDS]
    for _ in range(180):
        unit = (b"ab", b"\0a", b"abc", b"\0\0a")[int(rng.integers(0, 4))]
        w = b"".join(unit * int(rng.integers(2, 30)) + bytes([int(rng.choice(list(b"cdf\0")))]) * int(rng.integers(1, 3))
                     for _ in range(int(rng.integers(1, 4))))
        k = int(rng.integers(0, len(w)))
        blocks.append((w[k:] + w[:k]) * int(rng.integers(2, 13)))
    _bwt_equals_oracle(lfc, blocks)


def _frames(name):
    if name == "zero":  # RLE1: 255-byte pieces, all alike
        return [np.zeros((255, 255), np.uint16)], 15, (0, 0x14, 0x64)
    if name == "constant":
        return [np.full((45, 30), 0x1234, np.uint16)], 15, (0, 0x40)
    if name == "rows":
        return [np.tile(np.random.default_rng(3).integers(0, 4000, 1020).astype(np.uint16), (255, 1))], 15, (0, 0x40)
    if name == "runs":  # in blocks of 900 bytes most hold one two-byte value
        rng = np.random.default_rng(17)
        n = np.concatenate([np.arange(1, 300), [1000, 4095, 4096, 4097, 20000]])
        return [np.resize(np.repeat(rng.integers(0, 65536, n.size, dtype=np.uint16), n), (285, 285))], 15, (0, 0x40)
    # words of 2 .. 997 pixels over and over, next to noise
    rng = np.random.default_rng(19)
    out = [np.resize(rng.integers(0, 300, n).astype(np.uint16), 60 * n).reshape(60, n) for n in (2, 3, 64, 100, 997)]
    return [np.ascontiguousarray(f) for f in out] + [rng.integers(0, 65536, (60, 90), dtype=np.uint16)], 1, (0,)


def _decode(lfc, plan, blobs, shapes):
    import torch
    outs = [torch.zeros(s, dtype=torch.int16, device="cuda") for s in shapes]
    plan.decompress([torch.from_numpy(np.frombuffer(b, dtype=np.uint8).copy()).cuda() for b in blobs], outs)
    return [lfc.from_device_frame(o) for o in outs]


def test_repeated_blocks_form_several_cycles():
    """What the decoder meets: the origin's cycle is the repeated string, read
    backwards; stock bzip2 writes it until the block is full."""
    raw = _frames("constant")[0][0].tobytes()
    r = oracle.rle1(raw)
    L, orig = oracle.bwt(r)
    nxt, row, cyc = _rows(r.size, L), orig, []
    while not cyc or row != orig:
        cyc.append(int(L[row]))
        row = int(nxt[row])
    assert len(cyc) == 2 and r.size % 2 == 0
    assert bytes(r) == bytes(cyc[::-1]) * (r.size // 2)
    assert bz2.decompress(oracle.bz2_stream(raw)) == raw


@pytest.mark.gpu
@pytest.mark.parametrize("name,block_bytes", [("zero", 720000), ("zero", 900), ("constant", 720000), ("constant", 901),
                                              ("rows", 720000), ("rows", 65280), ("runs", 900), ("words", 720000)])
def test_repeated_blocks_decode(lfc, name, block_bytes):
    frames, p, ids = _frames(name)
    w, h = max(f.shape[1] for f in frames), max(f.shape[0] for f in frames)
    plan = lfc.Plan(w, h, p, max_frames=len(frames), block_bytes=block_bytes)
    for cid in ids:
        blobs = [oracle.compress_id(f, p, cid, block_bytes=block_bytes) for f in frames]
        for got, f in zip(_decode(lfc, plan, blobs, [f.shape for f in frames]), frames):
            assert np.array_equal(got, f)
    # judged and compressed here, then read back
    ds = [lfc.to_device_frame(f) for f in frames]
    blobs = plan.compress_to_bytes(ds, p)
    for got, f in zip(_decode(lfc, plan, blobs, [f.shape for f in frames]), frames):
        assert np.array_equal(got, f)
    plan.close()


@pytest.mark.gpu
def test_repeated_blocks_damaged(lfc):
    """Damage is refused or gives the exact frame."""
    fr = np.resize(np.random.default_rng(23).integers(0, 300, 24).astype(np.uint16), (40, 60))
    blob = oracle.compress_id(fr, 1, 0)
    plan = lfc.Plan(60, 40, 1)
    for bit in range(8 * 44 + 112, 8 * len(blob), 5):  # from the origin row on
        t = bytearray(blob)
        t[bit >> 3] ^= 0x80 >> (bit & 7)
        try:
            got = _decode(lfc, plan, [bytes(t)], [fr.shape])[0]
        except lfc.LfcError as e:
            assert e.status == 3, e
            continue
        assert np.array_equal(got, fr), bit
    plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(64, 1406), (256, 1020), (96, 1406), (48, 2000)])
def test_nearly_repeated_blocks_are_not_serial(lfc, shape):
    """One row over and over with one pixel changed: as fast as noise of the
    same size, give or take (a piece of 100 000 rows and more, walked by one
    thread, took over 20 times as long)."""
    import torch
    rng = np.random.default_rng(29)
    near = np.tile(rng.integers(0, 4096, shape[1]).astype(np.uint16), (shape[0], 1))
    near[-1, -1] ^= 1
    ms = []
    plan = lfc.Plan(shape[1], shape[0], 2)
    for fr in (near, rng.integers(0, 4096, shape).astype(np.uint16)):
        blob = torch.from_numpy(np.frombuffer(oracle.compress_id(fr, 2, 0), dtype=np.uint8).copy()).cuda()
        out = torch.zeros(shape, dtype=torch.int16, device="cuda")
        best = float("inf")
        for _ in range(3):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.decompress([blob], [out])
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert np.array_equal(lfc.from_device_frame(out), fr)
        ms.append(best)
    plan.close()
    assert ms[0] < 4 * ms[1], ms


def _skewed(rng, n):
    return np.minimum(rng.geometric(0.3, n), 255).astype(np.uint8).tobytes()


@pytest.mark.gpu
@pytest.mark.parametrize("copies", [2, 8, 32])
def test_long_repeats_encode(lfc, copies):
    """24 blocks of a string over and over (prefix doubling orders them) take
    no more than 8 times as long as 24 plain ones, and give the oracle's
    streams (walking every group of ties far took 14 times as long)."""
    import torch
    rng = np.random.default_rng(67)

    def repeats():
        w = _skewed(rng, 100000 // copies)
        return b"".join(w + _skewed(rng, 20) for _ in range(copies))

    plan = lfc.Plan(2040, 2040, 15, max_frames=2)
    ms = []
    for blocks in ([repeats() for _ in range(24)], [_skewed(rng, 100000) for _ in range(24)]):
        sizes = [len(b) for b in blocks]
        offs = [int(v) for v in np.cumsum([0] + sizes[:-1])]
        data = torch.from_numpy(np.frombuffer(b"".join(blocks), dtype=np.uint8).copy()).cuda()
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            out, n, stride = plan.bzip2_encode(data, offs, sizes)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        ms.append(best)
        out, n = out.cpu().numpy(), n.cpu().numpy()
        for i in (0, 11, 23):
            assert out[i * stride:i * stride + int(n[i])].tobytes() == oracle.bz2_stream(blocks[i]), i
    plan.close()
    assert ms[0] < 8 * ms[1], ms
