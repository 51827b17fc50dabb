"""Batches in which a refused field's last chunk and the next field's first one share a ticket: the
compression kernel has loaded the refused chunk's values before it knows of the refusal, and the next
chunk's go into the same buffer. The good fields' streams are the one-field call's, on every call."""
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHUNK = 8192


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


# (pairs of a refused and a good field, the good fields' chunks): tickets are two chunks from 2432
# chunks on, 304 of them are taken before the fields' steps are known. 64 fields are planned by the
# value-range kernel for itself, 200 by the planning kernel.
@pytest.mark.parametrize("pairs,chunks", [(32, 17), (100, 1)])
@pytest.mark.parametrize("ragged", [0, 5])
def test_a_refused_chunk_and_the_next_fields_first(fszlib, pairs, chunks, ragged):
    dev = _cuda()
    src = torch.from_numpy(inputs.sinusoids(1 << 20, seed=7)).to(dev)
    good = [src[64 * k:64 * k + chunks * CHUNK - ragged].clone() for k in range(pairs)]
    good[-1] = src.repeat(20)[:2500 * CHUNK - ragged].clone()
    refused = [torch.full((CHUNK - ragged,), 1e4, device=dev) for _ in range(pairs)]
    for k, x in enumerate(refused):
        x[37 * k % x.numel()] = float("nan")
    xs = [x for pair in zip(refused, good) for x in pair]
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    refs = [fszlib.compress(x, 1e-3)[0] for x in good]
    for _ in range(8):
        b.arena.fill_(0xA5)
        b.sizes.zero_()
        assert b.run() == fszlib.OK
        assert b.status()[1] == [fszlib.ERR_NONFINITE, fszlib.OK] * pairs
        ks = b.sizes.cpu().tolist()
        for k, ref in enumerate(refs):
            assert ks[2 * k] == 0 and ks[2 * k + 1] == ref.numel()
            assert torch.equal(b.stream(2 * k + 1, ks), ref), k
