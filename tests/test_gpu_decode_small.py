"""The decoder on blocks of every size: grids and segment counts follow the
largest block of the call. Frames come back exactly, a stream of more bytes
than its container promises is refused, and many small blocks do not cost what
as many large ones would."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lfc():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


def _dev(b):
    import torch
    return torch.from_numpy(np.frombuffer(b, dtype=np.uint8).copy()).cuda()


# a segment count is a multiple of 384 for every 12288 bytes of a block's last
# column (5/4 of the block), tiles have 4096 of them
@pytest.mark.parametrize("shape,block_bytes", [((15, 15), 1), ((15, 15), 7), ((30, 45), 100), ((45, 60), 3276), ((45, 60), 3277),
                                               ((150, 150), 9829), ((150, 150), 9830), ((150, 150), 9831), ((300, 300), 50000),
                                               ((300, 300), 86015), ((300, 300), 86017), ((300, 300), 180000)])
def test_block_sizes(lfc, shape, block_bytes):
    import torch
    rng = np.random.default_rng(block_bytes)
    frames = [rng.poisson(90, shape).astype(np.uint16), np.minimum(rng.geometric(0.7, shape), 9).astype(np.uint16),
              rng.integers(0, 65536, shape).astype(np.uint16)]
    frames.append(np.where(rng.random(shape) < 0.01, 700, 40).astype(np.uint16))
    plan = lfc.Plan(shape[1], shape[0], 15, max_frames=4, block_bytes=block_bytes)
    blobs = [oracle.compress_id(f, 15, cid, block_bytes=block_bytes) for f, cid in zip(frames, (0, 0x14, 0x40, 0x65))]
    outs = [torch.zeros(shape, dtype=torch.int16, device="cuda") for _ in frames]
    plan.decompress([_dev(b) for b in blobs], outs)
    for o, f in zip(outs, frames):
        assert np.array_equal(lfc.from_device_frame(o), f)
    plan.close()


@pytest.mark.parametrize("other", [(60, 60), (300, 300)])
def test_more_bytes_than_promised(lfc, other):
    """The stream of a larger frame in a smaller one's container."""
    import torch
    rng = np.random.default_rng(31)
    small = oracle.compress_id(rng.poisson(90, (30, 30)).astype(np.uint16), 15, 0)
    for big in (rng.poisson(90, other), np.full(other, 5), np.minimum(rng.geometric(0.9, other), 3)):
        s = oracle.compress_id(np.asarray(big, dtype=np.uint16), 15, 0)[44:]
        plan = lfc.Plan(300, 300, 15)
        out = torch.zeros((30, 30), dtype=torch.int16, device="cuda")
        with pytest.raises(lfc.LfcError) as e:
            plan.decompress([_dev(small[:40] + np.uint32(len(s)).tobytes() + s)], [out])
        assert e.value.status == 3
        plan.close()


def test_many_small_blocks(lfc):
    """338 blocks a frame take no more than 3.6 times as long as 16 (2.5 times
    where this was written; with grids for blocks of 720 000 bytes 4.5 times)."""
    import torch
    fr = np.random.default_rng(37).poisson(100, (390, 390)).astype(np.uint16)
    ms = []
    for block_bytes in (900, 20000):
        plan = lfc.Plan(390, 390, 13, max_frames=2, block_bytes=block_bytes)
        blobs = [_dev(b) for b in plan.compress_to_bytes([lfc.to_device_frame(fr)] * 2, 13)]
        outs = [torch.zeros(fr.shape, dtype=torch.int16, device="cuda") for _ in blobs]
        best = float("inf")
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            plan.decompress(blobs, outs)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        assert all(np.array_equal(lfc.from_device_frame(o), fr) for o in outs)
        ms.append(best)
        plan.close()
    assert ms[0] < 3.6 * ms[1], ms
