"""Quads of very different lengths side by side in a chunk (none, one block, exactly 128 or 256
words, and one word pair either side of that): the stream's runs against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

QUAD, CHUNK = 1024, 8192


def _quad(rate, blocks=32, extra=None):
    """Values 0, a, 0, a, .. in the first `blocks` blocks, a giving them `rate`; `extra`: the
    rate of the last of them."""
    x = np.zeros(QUAD)
    for b in range(blocks):
        r = extra if extra is not None and b == blocks - 1 else rate
        x[32 * b + 1:32 * b + 30:2] = 1 if r == 1 else 3 << max(r - 2, 0) if r else 0
    return x


@pytest.mark.parametrize("rotation", range(8))
@pytest.mark.parametrize("tail", [0, 1, 2500])
def test_runs_of_uneven_length(fszlib, oracle, rotation, tail):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    quads = [_quad(0), _quad(1, 1), _quad(3), _quad(3, extra=4), _quad(3, extra=2), _quad(7),
             _quad(15), _quad(7, extra=6)]
    chunk = np.concatenate([quads[(k + rotation) % 8] for k in range(8)])
    x = np.concatenate([chunk, chunk[::-1], np.tile(quads[2], 8), chunk[:tail]]).astype(np.float32)
    ref = np.frombuffer(oracle.compress(x, 0.47, oracle.ABS), np.uint8)
    sb, nb = fszlib.compress(torch.from_numpy(x).to("cuda:0"), 0.47, fszlib.EB_ABS)
    assert nb == ref.size and np.array_equal(sb.cpu().numpy(), ref)
    words = (ref[64:64 + 8 * (CHUNK // 256)] & 31).astype(int)   # the first chunk's rates
    words = np.where(words > 0, words + 1, 0).reshape(8, 32).sum(axis=1)
    assert sorted(words) == [0, 2, 127, 128, 129, 255, 256, 512]
