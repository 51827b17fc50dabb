"""Tiles whose sum overflows float32, in every tile configuration: partial sums of both signs that
overflow leave no mean (512- and 1024-element tiles), others an infinite one. Such a tile's centred
variants always lose, as in the oracle, whatever block 0 would save by them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CONFIGS = [(32, 4), (32, 8), (32, 16), (64, 4), (64, 8), (64, 16)]
A = np.float32(2.0 ** 120.38)  # near the largest magnitude that the step's cap of 2^101 admits


def _tile(size, block, kind):
    """Block 0 level, so that centring it would save its first residual; then waves whose even and
    odd 8-element runs have opposite signs (or one sign and zero), which is how the tile's last
    additions meet."""
    wave = {"square": [1, -1], "gaps": [1, 0, -1, 0], "one_sign": [1, 1], "halves": [1, 0]}[kind]
    x = np.resize(np.repeat(np.array(wave, np.float32), 8), size)
    x[:block] = 1
    return A * x


@pytest.mark.parametrize("B,T", CONFIGS)
@pytest.mark.parametrize("sign", [1, -1])
def test_tiles_without_a_finite_mean(fszlib, oracle, B, T, sign):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    rng = np.random.default_rng(B * T)
    tiles = [_tile(B * T, B, kind) for kind in ("square", "gaps", "one_sign", "halves")]
    tiles += [(A * rng.uniform(-1, 1, B * T)).astype(np.float32), np.full(B * T, A / 2, np.float32)]
    x = (sign * np.concatenate(tiles * 9 + [tiles[0][:B * T // 2 + 5]])).astype(np.float32)
    ref = oracle.compress_cfg(x, 1e-3, oracle.REL, B, T)
    xd = torch.from_numpy(x).cuda()
    sb, nb = fszlib.compress_tiled(xd, 1e-3, fszlib.EB_REL, B, T)
    assert sb.cpu().numpy().tobytes() == ref
    y = fszlib.decompress_tiled(sb, x.size).cpu().numpy()
    assert np.array_equal(y.view(np.uint32), oracle.decompress(ref).view(np.uint32))
    if (B, T) == (32, 8):
        assert fszlib.compress(xd, 1e-3)[0].cpu().numpy().tobytes() == ref
        b = fszlib.CompressBatch([(xd, (x.size,), fszlib.EB_REL, 1e-3)] * 2, device="cuda")
        assert b.run() == fszlib.OK and torch.equal(b.stream(1), sb)
