"""fsz_decompress_tiled on damaged streams: rate headers with reserved or switched-off bits, or whose
sizes do not add up to the preamble's, are found before anything is decoded, so the output is left as
it was, wherever in the stream the damage is."""
import numpy as np
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CONFIGS = [(32, 4), (32, 8), (32, 16), (64, 4), (64, 8), (64, 16)]
CHUNK = 8192


def _damaged(s, B, T, n, off):
    """(what, bytes) of streams that differ from the good one s in a header or the data's size."""
    NT = -(-n // (B * T))
    db = int(s[56:64].view(np.uint64)[0])

    def at(pos, change):
        bad = s.copy()
        bad[pos] = change(int(bad[pos]))
        return bad

    def size(d):
        bad = s.copy()
        bad[56:64] = np.frombuffer(np.uint64(db + d).tobytes(), np.uint8)
        return bad

    for t in (0, NT // 2, NT - 1):         # a tile of the first chunk, one between, the last one
        first = 64 + T * t
        yield f"reserved bit 5 of tile {t}", at(first, lambda v: v | 0x20)
        yield f"reserved bit 6 of tile {t}'s second block", at(first + 1, lambda v: v | 0x40)
        yield f"a plane more in tile {t}", at(first + T - 1, lambda v: (v & 0xE0) | ((v & 31) + 1) % 32)
        yield f"a mean more or less in tile {t}", at(first, lambda v: v ^ 0x40)
        if off:
            yield f"a switched-off feature in tile {t}", at(first, lambda v: v | 0x80)
    yield "4 bytes less declared", size(-4)
    if s.size - 64 - T * NT - db >= 4:
        yield "4 bytes more declared", size(4)


def _decompress(fszlib, stream, out):
    src = torch.from_numpy(stream).to(out.device)
    wsb = fszlib.lib().fsz_tiled_workspace_bytes(out.numel())
    ws = torch.full((wsb,), 0xFF, dtype=torch.uint8, device=out.device)
    sp = torch.cuda.current_stream().cuda_stream
    assert fszlib.lib().fsz_decompress_tiled(src.data_ptr(), src.numel(), out.data_ptr(), out.numel(),
                                             ws.data_ptr(), wsb, sp) == fszlib.OK
    return fszlib.fsz_check(ws.data_ptr(), sp)


@pytest.mark.parametrize("B,T", CONFIGS)
@pytest.mark.parametrize("n,off", [(40 * CHUNK + 5, 0), (700 * CHUNK - 3, 0), (3 * CHUNK, 4)])
def test_a_damaged_stream_leaves_the_output_alone(fszlib, oracle, B, T, n, off):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    x = np.resize(inputs.sinusoids(1 << 18, seed=3), n)
    ref = np.frombuffer(oracle.compress_cfg(x, 1e-3, oracle.REL, B, T, off), np.uint8)
    s = np.concatenate([ref, np.zeros(16, np.uint8)])    # room behind the stream
    out = torch.full((n,), 7.0, dtype=torch.float32, device=dev)
    for what, bad in _damaged(s, B, T, n, off):
        assert _decompress(fszlib, bad, out) == fszlib.ERR_CORRUPT, what
        assert bool((out == 7.0).all()), what
    assert _decompress(fszlib, s, out) == fszlib.OK
    assert np.array_equal(out.cpu().numpy().view(np.uint32), oracle.decompress(ref.tobytes()).view(np.uint32))
