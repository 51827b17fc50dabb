"""Tile configurations at the edges of tiles, header units, quads and chunks, over every
feature set that the format allows, and their damaged streams, against the oracle."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CONFIGS = [(32, 4), (32, 8), (32, 16), (64, 4), (64, 8), (64, 16)]
CHUNK = 8192


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _field(n, seed):
    """Offsets that change by tile (centred and uncentred tiles side by side), ramps (second
    order) and noise of changing scale."""
    rng = np.random.default_rng(seed)
    k = -(-n // 96)
    off = np.repeat(rng.choice([0.0, 0.0, 50.0, -300.0], k), 96)[:n]
    scale = np.repeat(10.0 ** rng.uniform(-4, 0.5, k), 96)[:n]
    ramp = np.cumsum(np.repeat(rng.choice([0.0, 0.02, 2.0, -2.0], k), 96)[:n])
    return (off + ramp + scale * rng.standard_normal(n)).astype(np.float32)


@pytest.mark.parametrize("off", [0, 2, 4, 6, 3, 7])
@pytest.mark.parametrize("B,T", CONFIGS)
def test_edges_and_features(fszlib, oracle, B, T, off):
    dev = _cuda()
    tile = B * T
    sizes = {1, 31, 33, tile - 1, tile, tile + 1, 2 * tile + 1, 3 * tile, 1024 - 1, 1024 + 1,
             CHUNK - tile, CHUNK - 1, CHUNK + 1, 3 * CHUNK + tile, 33 * CHUNK + 5 * tile + 7}
    for n in sorted(sizes):
        x = _field(n, n + off)
        ref = oracle.compress_cfg(x, 0.05, oracle.ABS, B, T, off)
        sb, _ = fszlib.compress_tiled(torch.from_numpy(x).to(dev), 0.05, fszlib.EB_ABS, B, T, off)
        assert sb.cpu().numpy().tobytes() == ref, n
        y = fszlib.decompress_tiled(sb, n).cpu().numpy()
        assert np.array_equal(y.view(np.uint32), oracle.decompress(ref).view(np.uint32)), n


@pytest.mark.parametrize("B,T", CONFIGS)
def test_damaged_streams(fszlib, oracle, B, T):
    dev = _cuda()
    n = 3 * CHUNK + 5 * B * T + 7
    s = np.frombuffer(oracle.compress_cfg(_field(n, 1), 0.05, oracle.ABS, B, T, 0), np.uint8)
    NT = -(-n // (B * T))
    hdr = slice(64, 64 + T * NT)

    def status(buf):
        try:
            fszlib.decompress_tiled(torch.from_numpy(buf).to(dev), n)
        except fszlib.FszError as e:
            return e.status
        return fszlib.OK

    assert status(s.copy()) == fszlib.OK
    for at, bit in ((64, 0x20), (64 + T, 0x20), (64 + 1, 0x40), (64 + T * (NT - 1) + T - 1, 0x80),
                    (64 + T + 2, 0x20), (53, 0x40), (53, 0x04), (54, 0x01)):
        bad = s.copy()
        bad[at] ^= bit
        assert status(bad) == fszlib.ERR_CORRUPT, (at, bit)
    bad = s.copy()
    bad[hdr][-1] ^= 1                       # a rate that moves the total by one word
    assert status(bad) == fszlib.ERR_CORRUPT
    assert status(s[:-16].copy()) == fszlib.ERR_CORRUPT
    centred = np.nonzero(s[64:64 + T * NT:T] & 0x40)[0]
    if centred.size:                        # a mean that is no integer
        rates = (s[hdr] & 31).reshape(NT, T).astype(np.int64)
        size = np.where(rates > 0, (B // 8) * (rates + 1), 0).sum(1) + np.where(s[64:64 + T * NT:T] & 0x40, 4, 0)
        at = 64 + T * NT + int(size[:centred[-1]].sum())
        bad = s.copy()
        bad[at:at + 4] = np.frombuffer(np.float32(0.5).tobytes(), np.uint8)
        assert status(bad) == fszlib.ERR_CORRUPT
