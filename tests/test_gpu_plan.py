"""Batch planning across its 1024-field rounds: streams, sizes, statuses and reconstructions of
each field equal the one-field call's, in a workspace full of another batch's leftovers."""
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("nfields", [1, 2, 31, 33, 1023, 1024, 1025, 2049])
def test_batches_of_many_fields(fszlib, nfields):
    dev = _cuda()
    src = torch.from_numpy(inputs.sinusoids(1 << 17, seed=3)).to(dev)
    # empty fields, single tiles, chunks and a few long ones
    sizes = [(0, 1, 255, 257, 700, 8191, 8193)[k % 7] + (20000 if k % 97 == 5 else 0) for k in range(nfields)]
    xs = [src[64 * (k % 700):64 * (k % 700) + n].clone() for k, n in enumerate(sizes)]
    refused = {k for k in range(nfields) if k % 41 == 9 and sizes[k]}
    for k in refused:
        xs[k][sizes[k] // 2] = float("nan")
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    b.ws.fill_(0xFF)                       # leftovers in every word of the workspace
    assert b.run() == fszlib.OK
    st, per = b.status()
    assert per == [fszlib.ERR_NONFINITE if k in refused else fszlib.OK for k in range(nfields)]
    assert st == (fszlib.ERR_NONFINITE if refused else fszlib.OK)
    ks = b.sizes.cpu().tolist()
    keep = [k for k in range(nfields) if k not in refused]
    check = keep if nfields < 100 else keep[:20] + keep[len(keep) // 2:len(keep) // 2 + 20] + keep[-30:]
    for k in check:
        ref, nb = fszlib.compress(xs[k], 1e-3)
        assert ks[k] == nb and torch.equal(b.stream(k, ks), ref), k
    d = fszlib.DecompressBatch([b.stream(k, ks) for k in keep], [sizes[k] for k in keep], device=dev)
    d.ws.fill_(0xFF)
    assert d.run() == fszlib.OK
    assert d.status() == (fszlib.OK, [fszlib.OK] * len(keep))
    for i, k in enumerate(keep):
        if k in check:
            assert torch.equal(d.output(i), fszlib.decompress(b.stream(k, ks), n=sizes[k])), k
