"""Blocks that repeat a shorter string: the origin row among identical
rotations."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


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
