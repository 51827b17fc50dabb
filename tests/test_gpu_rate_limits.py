"""The rates at the top of the range, 21 to 23: steep ramps, which the second order takes for little,
around one block of full-scale swings, whose second-order residuals reach 2^22."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILE, EB = 256, 0.5
A = 1_398_000 * EB  # near the second margin tier's limit


def ramps_and_swings(block, slope_sign):
    """A tile that ramps up to +-A before `block`, swings between A and -A in it, and ramps on."""
    x = np.empty(TILE)
    lo, hi = 32 * block, 32 * block + 32
    x[:lo] = np.linspace(-A, A, lo, endpoint=False) if lo else []
    x[lo:hi] = np.where(np.arange(32) % 2 == 0, A, -A)
    x[hi:] = np.linspace(-A, A, TILE - hi) if hi < TILE else []
    return slope_sign * np.rint(x)


def field(seed):
    rng = np.random.default_rng(seed)
    tiles = [ramps_and_swings(b, s) for b in range(8) for s in (1, -1)]
    tiles += [rng.integers(-(1 << k), (1 << k) + 1, TILE) * EB for k in range(19, 21)]
    tiles += [np.cumsum(rng.integers(-2, 3, TILE)) * 1.0, np.zeros(TILE)]
    order = rng.permutation(np.repeat(np.arange(len(tiles)), 24))
    return np.concatenate([tiles[k] for k in order])[:-3].astype(np.float32)


@pytest.mark.parametrize("seed", [0, 1])
def test_the_top_rates(fszlib, oracle, seed):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    x = field(seed)
    ref = oracle.compress(x, EB, oracle.ABS)
    want = np.frombuffer(ref, np.uint8)
    hdr = want[64:64 + 8 * -(-x.size // TILE)].reshape(-1, 8)
    assert set(range(21, 24)) <= set(int(r) for r in hdr.ravel() & 31)
    assert ((hdr[:, 0] & 0x80 != 0) & ((hdr & 31).max(1) == 23)).any()
    xd = torch.from_numpy(x).cuda()
    sb, nb = fszlib.compress(xd, EB, fszlib.EB_ABS)
    assert nb == want.size and sb.cpu().numpy().tobytes() == ref
    y = fszlib.decompress(sb, n=x.size).cpu().numpy()
    assert np.array_equal(y.view(np.uint32), oracle.decompress(ref).view(np.uint32))
    for B, T in ((32, 4), (32, 16), (64, 4), (64, 16)):
        r = oracle.compress_cfg(x, EB, oracle.ABS, B, T)
        s, _ = fszlib.compress_tiled(xd, EB, fszlib.EB_ABS, B, T)
        assert s.cpu().numpy().tobytes() == r, (B, T)
        y = fszlib.decompress_tiled(s, x.size).cpu().numpy()
        assert np.array_equal(y.view(np.uint32), oracle.decompress(r).view(np.uint32)), (B, T)
