"""The bit-sliced census of the fixed windows at the edges of its units (128 columns x 32
rows), its four words a row, its 16-byte and word loads: widths and heights around multiples,
row pitches and base addresses of every alignment, the last row ending with its buffer."""
import numpy as np
import pytest

from oracle import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3])
@pytest.mark.parametrize("W,H", [(1, 40), (4, 7), (31, 33), (127, 31), (128, 32), (129, 33), (131, 64), (133, 65),
                                 (255, 35), (256, 8), (260, 38), (516, 97)])
def test_unit_edges_equal_oracle(W, H, k):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    rng = np.random.default_rng(1000 * W + 10 * H + k)
    for pad, base in ((0, 0), (0, 5), (3, 2), (16 - W % 16, 0), (4 - W % 4, 8)):
        pitch = W + pad
        buf = torch.from_numpy(rng.integers(0, 256, base + pitch * (H - 1) + W, dtype=np.uint8)).cuda()
        buf[base:base + pitch * (H // 3)] = 90  # ties
        img = buf[base:].as_strided((H, W), (pitch, 1))
        host = np.ascontiguousarray(img.cpu().numpy())
        for win in ((9, 7), (7, 7), (5, 5)):
            got = B.census_build(img, k, *win, 1).cpu().numpy().view(np.uint64)
            ref = orc.census(host, k, *win, 1)
            assert np.array_equal(got, ref), (pad, base, win, np.argwhere(got != ref)[:5].tolist())
