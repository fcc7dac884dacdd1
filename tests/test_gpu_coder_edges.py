"""The entropy coder's and the judge's choices by size: MTF segments of 1024
and 4096 bytes, the chain walk's shortest ranges, CRC pieces at every
alignment, code lengths cut to 17 bits, odd tile widths of the emission.
Streams and scores equal the oracle's."""
import bz2

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lfc():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


def _encode(lfc, plan, blocks):
    import torch
    data = torch.from_numpy(np.frombuffer(b"".join(blocks), dtype=np.uint8).copy()).cuda()
    sizes = [len(b) for b in blocks]
    offs = [int(v) for v in np.cumsum([0] + sizes[:-1])]
    stride = lfc.max_stream_bytes(max(sizes))
    out, n = plan.bzip2_encode(data, offs, sizes, stride=stride)[:2]
    out, n = out.cpu().numpy(), n.cpu().numpy()
    return [out[i * stride:i * stride + int(n[i])].tobytes() for i in range(len(blocks))]


def test_streams_equal_oracle(lfc):
    rng = np.random.default_rng(41)
    blocks = [bytes(rng.integers(0, 40, n, dtype=np.uint8)) for n in
              (1, 2, 15, 16, 17, 31, 1023, 1024, 1025, 2049, 4095, 4096, 4097, 8191, 12289, 16383, 16385, 65537)]
    # ranks of probability 2^-k: codes of more than 17 bits before the cut
    blocks.append(bytes(np.minimum(rng.geometric(0.5, 700001), 255).astype(np.uint8)))
    blocks.append(bytes(rng.integers(0, 256, 100003, dtype=np.uint8)))
    blocks += [b"\x07" * 50000, b"ab" * 3000 + b"b"]
    plan = lfc.Plan(2040, 2040, 15, max_frames=2)
    for i, (got, b) in enumerate(zip(_encode(lfc, plan, blocks), blocks)):
        assert got == oracle.bz2_stream(b), i
        assert bz2.decompress(got) == b, i


def test_mtf_segment_lengths(lfc):
    """Above about 40 MB of blocks the MTF segments have 4096 bytes, below it
    1024: the same blocks on both sides of the line give the same streams."""
    rng = np.random.default_rng(43)
    base = [bytes(np.minimum(rng.geometric(0.1, 720000), 255).astype(np.uint8)) for _ in range(3)]
    blocks = [base[i % 3] for i in range(60)]
    plan = lfc.Plan(2040, 2040, 15, max_frames=6)
    few, many = _encode(lfc, plan, blocks[:12]), _encode(lfc, plan, blocks)
    assert all(many[i] == few[i % 3] for i in range(60))
    for i in range(3):
        assert few[i] == oracle.bz2_stream(base[i])


@pytest.mark.parametrize("frames,p", [([(3, 3)], 3), ([(15, 30)], 15), ([(26, 39), (130, 13), (65, 65)], 13),
                                      ([(120, 120)] * 7, 15), ([(400, 390)], 10), ([(56, 112), (48, 64)], 8),
                                      ([(122, 183)], 61)])
def test_judge_small(lfc, frames, p):
    rng = np.random.default_rng(47)
    fr = [rng.poisson(90, f).astype(np.uint16) for f in frames]
    ids = oracle.default_ids()
    w, area = max(f[1] for f in frames), max(f[0] * f[1] for f in frames)
    plan = lfc.Plan(w, p * -(-area // (w * p)), p, max_frames=len(fr))
    choice, scores = plan.judge([lfc.to_device_frame(f) for f in fr], p)
    got = scores.cpu().numpy().view(np.uint64)
    for i, f in enumerate(fr):
        best, ref = oracle.judge(f, p, ids)
        assert [int(got[i][c]) for c in ids] == ref, i
        assert int(choice[i]) == best


def test_judge_all_functions_and_layouts(lfc):
    """Candidate sets other than the default: every function, both layouts."""
    rng = np.random.default_rng(53)
    ids = sorted({oracle.make_id(f, d, o, 0, pl) for f in range(1, 8) for d in range(3) for o in (0, 1) for pl in (0, 1)})
    for shape, p in (((48, 96), 6), ((45, 75), 5)):
        fr = rng.integers(0, 65536, shape).astype(np.uint16)
        plan = lfc.Plan(shape[1], shape[0], p, candidate_ids=ids)
        _, scores = plan.judge([lfc.to_device_frame(fr)], p)
        _, ref = oracle.judge(fr, p, ids)
        got = scores.cpu().numpy().view(np.uint64)[0]
        assert [int(got[c]) for c in ids] == ref, shape
