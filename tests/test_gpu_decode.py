"""The decoder where its parallel stages can go wrong: Huffman codes longer
than its lookups (and groups too long for its tables of 50-code lengths),
blocks of fewer symbols than it has segments, runs across segment and tile
edges, more blocks than one batch of frames, a lenslet grid too large for
shared memory. Frames equal what was encoded; damaged streams are refused or
give the exact frame."""
import bz2

import numpy as np
import pytest

import oracle


def _stream(raw, lens):
    """The one-block bzip2 stream of raw with two code tables of the given
    lengths (functions of the symbol count) used in turn."""
    r = oracle.rle1(raw)
    L, orig = oracle.bwt(r)
    sym, in_use, _ = oracle.mtf_rle2(L)
    alpha = int(in_use.sum()) + 2
    bits = []

    def put(v, n):
        bits.append(format(int(v), "0%db" % n))

    for c in b"BZh9":
        put(c, 8)
    put(0x314159265359, 48)
    crc = oracle.crc32(raw)
    put(crc, 32)
    put(0, 1)
    put(orig, 24)
    used = in_use.reshape(16, 16)
    put(int("".join("1" if u.any() else "0" for u in used), 2), 16)
    for u in used:
        if u.any():
            put(int("".join("1" if x else "0" for x in u), 2), 16)
    nsel = -(-len(sym) // 50)
    put(2, 3)
    put(nsel, 15)
    bits.append("0" + "10" * (nsel - 1))  # tables 0, 1, 0, 1, ...: position 1 of the list after the first
    codes = []
    for f in lens:
        ln = f(alpha)
        put(ln[0], 5)
        cur, code, table = ln[0], 0, {}
        for x in ln:
            bits.append("10" * max(0, x - cur) + "11" * max(0, cur - x) + "0")
            cur = x
        for k in range(1, 21):
            for s, x in enumerate(ln):
                if x == k:
                    table[s] = format(code, "0%db" % k)
                    code += 1
            code <<= 1
        codes.append(table)
    for i in range(0, len(sym), 50):
        t = codes[(i // 50) & 1]
        bits.extend(t[int(s)] for s in sym[i:i + 50])
    put(0x177245385090, 48)
    put(crc, 32)
    b = "".join(bits)
    b += "0" * (-len(b) % 8)
    return int(b, 2).to_bytes(len(b) // 8, "big")


def _even(n):  # all codes of one length
    return lambda alpha: [n] * alpha


def _steps(alpha):  # 1, 2, 3, ... bits, the rest 20
    return [min(k + 1, 20) if k < 19 else 20 for k in range(alpha)]


CODES = {"9": [_even(9), _even(9)], "12": [_even(12), _even(12)], "13": [_even(13), _even(13)],
         "15_16": [_even(15), _even(16)],  # 8 codes of 120 and of 128 bits: the table's limit is 127
         "20": [_even(20), _even(20)], "steps_20": [_steps, _even(20)]}


def _recoded(name):
    fr = np.minimum(np.random.default_rng(5).geometric(0.4, (60, 90)), 17).astype(np.uint16)
    ref = oracle.compress_id(fr, 15, 0)
    s = _stream(fr.tobytes(), CODES[name])
    return fr, s, ref[:40] + np.uint32(len(s)).tobytes() + s


@pytest.mark.parametrize("name", list(CODES))
def test_recoded_streams_are_bzip2(name):
    fr, s, blob = _recoded(name)
    assert bz2.decompress(s) == fr.tobytes()
    assert np.array_equal(oracle.decompress(blob), fr)


@pytest.fixture(scope="module")
def lfc():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


def _decode(lfc, plan, blobs, frames):
    import torch
    outs = [torch.zeros(f.shape, dtype=torch.int16, device="cuda") for f in frames]
    plan.decompress([torch.from_numpy(np.frombuffer(b, dtype=np.uint8).copy()).cuda() for b in blobs], outs)
    for i, (o, f) in enumerate(zip(outs, frames)):
        assert np.array_equal(lfc.from_device_frame(o), f), i


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(CODES))
def test_long_codes(lfc, name):
    fr, _, blob = _recoded(name)
    _decode(lfc, lfc.Plan(90, 60, 15), [blob], [fr])


@pytest.mark.gpu
@pytest.mark.parametrize("name", list(CODES))
def test_long_codes_damaged(lfc, name):
    """A damaged stream is refused or gives the exact frame (every wait of the
    decoder is a barrier, every access bounds-checked)."""
    import torch
    fr, _, blob = _recoded(name)
    plan = lfc.Plan(90, 60, 15)
    rng = np.random.default_rng(11)
    for pos in rng.integers(44, len(blob), 12):
        t = bytearray(blob)
        t[pos] ^= 1 << int(rng.integers(0, 8))
        out = torch.zeros(fr.shape, dtype=torch.int16, device="cuda")
        try:
            plan.decompress([torch.from_numpy(np.frombuffer(bytes(t), dtype=np.uint8).copy()).cuda()], [out])
        except lfc.LfcError as e:
            assert e.status in (1, 2, 3), e
            continue
        assert np.array_equal(lfc.from_device_frame(out), fr), pos


def _content(name):
    rng = np.random.default_rng(17)
    if name == "one_lenslet":
        return [rng.integers(0, 65536, (3, 3), dtype=np.uint16)], 3, (0, 0x64)
    if name == "constant":
        return [np.full((300, 300), 0x0101, dtype=np.uint16)], 15, (0, 0x15)
    if name == "noise":  # every byte value, codes of equal length
        return [rng.integers(0, 65536, (195, 195), dtype=np.uint16)], 13, (0, 0x44)
    if name == "runs":  # constant stretches of 1 .. 20000 pixels: RLE1 counts and RUNA / RUNB runs of every length
        n = np.concatenate([np.arange(1, 300), [1000, 4095, 4096, 4097, 20000]])
        v = np.repeat(rng.integers(0, 65536, n.size, dtype=np.uint16), n)
        return [np.resize(v, (285, 285))], 15, (0, 0x40)
    if name == "grid":  # 102 720 lenslets: the view's grid does not fit shared memory
        return [rng.poisson(40, (963, 960)).astype(np.uint16)], 3, (0x14, 0x65)
    # more frames and geometries in one call than a batch of predictors takes
    return [rng.poisson(30 + k, (15 * (1 + k % 4), 15 * (1 + k % 3))).astype(np.uint16) for k in range(40)], 15, (0x14, 0x26)


# Not "runs" in blocks of 900 bytes: a block that repeats a shorter string
# (here two bytes) is refused, its rows form several cycles.
# (It was refused when this was written; test_gpu_repeats.py decodes such blocks.)
@pytest.mark.gpu
@pytest.mark.parametrize("name,block_bytes", [("one_lenslet", 900), ("one_lenslet", 720000), ("constant", 900),
                                              ("constant", 720000), ("noise", 900), ("noise", 720000), ("runs", 720000),
                                              ("grid", 100000), ("grid", 720000), ("many_frames", 900),
                                              ("many_frames", 720000)])
def test_contents(lfc, name, block_bytes):
    frames, p, ids = _content(name)
    w, h = max(f.shape[1] for f in frames), max(f.shape[0] for f in frames)
    plan = lfc.Plan(w, h, p, max_frames=len(frames), block_bytes=block_bytes)
    for cid in ids:
        _decode(lfc, plan, [oracle.compress_id(f, p, cid, block_bytes=block_bytes) for f in frames], frames)
