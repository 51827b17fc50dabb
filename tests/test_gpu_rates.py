"""Every rate from 0 to 23 and both sides of each power of two, with every sign pattern at
the ends of a block, through compression and decompression against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TILE = 256


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _field(order, seed, top):
    """Tiles of integers whose residuals reach just below, at and above 2^k (k up to `top`):
    level runs with one or two jumps, alternating signs, and uniform values."""
    rng = np.random.default_rng(seed)
    tiles = []
    for k in range(top + 1):
        for off in (-1, 0, 1):
            a = max(0, (1 << k) + off)
            jump = np.zeros(TILE)
            jump[rng.integers(0, TILE):] = a             # one LZ1 residual of exactly a
            drop = -jump
            spike = np.zeros(TILE)
            spike[32 * rng.integers(0, 8) + rng.choice([0, 1, 30, 31])] = -a
            alt = np.where(np.arange(TILE) % 2 == 0, a // 2, -(a - a // 2))
            uni = rng.integers(-a, a + 1, TILE)
            ramp = np.cumsum(rng.integers(-1, 2, TILE)) + a   # offset: centred variants
            tiles += [jump, drop, spike, alt, uni, ramp]
    if order == "mixed":
        rng.shuffle(tiles)
    return np.concatenate(tiles).astype(np.float32)


def _parity(fszlib, oracle, x, eb):
    dev = _cuda()
    ref = oracle.compress(x, eb, oracle.ABS)
    sb, nb = fszlib.compress(torch.from_numpy(x).to(dev), eb, fszlib.EB_ABS)
    got = np.frombuffer(sb.cpu().numpy().tobytes(), np.uint8)
    want = np.frombuffer(ref, np.uint8)
    assert nb == want.size and np.array_equal(got, want)
    y = fszlib.decompress(sb, n=x.size).cpu().numpy()
    assert np.array_equal(y.view(np.uint32), oracle.decompress(ref).view(np.uint32))
    T = -(-x.size // TILE)
    return set(int(r) for r in (want[64:64 + 8 * T] & 31))


@pytest.mark.parametrize("order", ["rising", "mixed"])
@pytest.mark.parametrize("top,eb,reach", [(4, 0.49, 5), (9, 0.49, 9), (16, 0.47, 17), (20, 0.76, 21)])
def test_every_rate(fszlib, oracle, order, top, eb, reach):
    # values up to 2^top in units of about one step; 2^20 needs the second margin tier
    rates = _parity(fszlib, oracle, _field(order, top, top), eb)
    assert set(range(0, min(reach, top) + 1)) <= rates


def test_the_largest_rate(fszlib, oracle):
    """Full-scale swings at the margin's limit: first-order residuals of rate 22."""
    a = 1_398_000 * 0.5
    x = np.where(np.arange(8 * TILE) % 2 == 0, a, -a).astype(np.float32)
    x[TILE:2 * TILE] = np.tile([a, a, -a, -a], TILE // 4)
    rates = _parity(fszlib, oracle, x, 0.5)
    assert max(rates) == 22
