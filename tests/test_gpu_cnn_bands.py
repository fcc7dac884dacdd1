"""The weight gradient's bands of rows (2, 4, 8 or 16, by the batch): every
gradient element against the fp64 oracle, at the bound of test_gpu_cnn.py, for
batches that take each height on a part of 152 SMs. The batches are powers of
two: the library divides by the batch before the pre-activation gradients are
rounded to BF16, the oracle after, and only then are the roundings the same."""
import numpy as np
import pytest

from oracle import cnn as ocnn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    from paper_2310_09467_gb300 import build, lfc
    build.build()
    return lfc


@pytest.fixture(scope="module")
def frames():
    """Three thumbnails with labels, and their gradients."""
    rng = np.random.default_rng(71)
    P = ocnn.init_params(32, 26, seed=71)
    for k in P:
        if k.startswith("b"):
            P[k] = 0.05 * rng.normal(size=P[k].shape)
    x = np.zeros((3, 2, 256, 256))
    x[:, :, :220, :243] = rng.uniform(0, 1.2, size=(3, 2, 220, 243))
    labels = [3, 17, 25]
    Pr = {k: (ocnn.bf16(v) if k.startswith("w") and k != "wl" else v) for k, v in P.items()}
    return P, x, labels, [ocnn.backward(Pr, ocnn.bf16(x[b]), labels[b], ocnn.bf16) for b in range(3)]


@pytest.mark.parametrize("n", [1, 4, 8, 32])
def test_gradients_match_oracle(L, frames, n):
    import torch
    P, x, labels, G = frames
    pick = np.random.default_rng(n).integers(0, 3, n)
    net = L.Cnn(26, n)
    net.set_params(net.flat_from_dict(P))
    net.set_thumbnails(torch.from_numpy(x[pick].astype(np.float32)).cuda())
    net.backward(torch.tensor([labels[k] for k in pick], dtype=torch.int32, device="cuda"))
    got = net.dict_from_flat(net.get_params(grads=True)[1])
    for k in G[0]:
        r = sum(G[b][k] for b in pick) / n
        bound = 1e-2 * np.abs(r) + 1e-3 * np.abs(r).max()
        err = np.abs(got[k] - r)
        worst = int(np.argmax(err / bound))
        assert np.all(err <= bound), (k, n, int((err > bound).sum()), float(err.flat[worst]), float(r.flat[worst]))
