"""Decompression of batches on both sides of the limits (512 fields; fields times CTAs) up to which
the sizing kernel plans for itself, with refused streams among them: statuses and values are the
one-field call's."""
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nfields,times", [(1, 1), (32, 1), (511, 1), (512, 1), (513, 1), (700, 1),
                                           (240, 24), (320, 24)])
def test_refused_streams_among_good_ones(fszlib, nfields, times):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    src = torch.from_numpy(inputs.sinusoids(1 << 20, seed=5)).to(dev)
    sizes = [times * (1, 8192, 300, 0, 8193, 16384, 40000)[k % 7] for k in range(nfields)]
    made = {n: fszlib.compress(src[:n].clone(), 1e-3)[0].clone() for n in set(sizes)}
    streams, caps, want = [], [], []
    for k, n in enumerate(sizes):
        s, cap, st = made[n].clone(), n, fszlib.OK
        if k % 9 == 3:
            s[0] ^= 1                                    # the magic
            st = fszlib.ERR_CORRUPT
        elif k % 9 == 5 and n > 8:
            cap, st = n - 5, fszlib.ERR_CAPACITY         # no room for the last elements
        elif k % 9 == 7 and n > 256:
            s, st = s[:64].clone(), fszlib.ERR_CORRUPT   # the headers cut off
        streams.append(s)
        caps.append(cap)
        want.append(st)
    d = fszlib.DecompressBatch(streams, caps, device=dev)
    d.ws.fill_(0xFF)
    assert d.run() == fszlib.OK
    status, per = d.status()
    assert per == want
    assert (status == fszlib.OK) == all(w == fszlib.OK for w in want)
    for k in [k for k in range(nfields) if want[k] == fszlib.OK][::max(1, nfields // 40)]:
        assert torch.equal(d.output(k), fszlib.decompress(made[sizes[k]], n=sizes[k])), k


def test_more_chunks_than_the_workspace_holds(fszlib):
    """The total over the slots: nothing is decoded, whichever kernel counts."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    x = torch.from_numpy(inputs.sinusoids(1 << 18, seed=6)).to(dev)
    s = fszlib.compress(x, 1e-3)[0].clone()
    d = fszlib.DecompressBatch([s] * 3, [x.numel()] * 3, device=dev)
    d.arena.fill_(0)
    sp = torch.cuda.current_stream().cuda_stream
    # a workspace for far fewer elements than the streams hold
    few = fszlib.lib().fsz_batch_workspace_bytes(8192, 3)
    assert fszlib.lib().fsz_decompress_batched(d.table.data_ptr(), 3, 8192, d.ws.data_ptr(), few, sp) == fszlib.OK
    assert fszlib.fsz_check(d.ws.data_ptr(), sp) == fszlib.ERR_WORKSPACE
    assert int(torch.count_nonzero(d.arena)) == 0
