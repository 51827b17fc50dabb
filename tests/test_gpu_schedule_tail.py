"""Decompression's tickets near a launch's end: at most 2 chunks, unless the schedule keeps the
requested size at every launch size (min_tickets_per_cta = 0)."""
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHUNK = 8192


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("ticket", [1, 2, 3, 4])
def test_a_held_schedule_keeps_its_tickets(fszlib, ticket, batch):
    """A chunk that is never handed over takes the rest of its ticket with it: with the first one
    held back, the output shows how many chunks the first ticket had."""
    dev = _cuda()
    n = 12 * CHUNK
    x = torch.from_numpy(inputs.sinusoids(n, seed=2)).to(dev)
    s = fszlib.compress(x, 1e-3)[0].clone()
    want = fszlib.decompress(s, n=n).clone()
    d = fszlib.DecompressBatch([s], [n], device=dev)
    out = d.arena[:n]
    out.fill_(7.0)
    ws = fszlib.Workspace(n, dev)
    sp = torch.cuda.current_stream().cuda_stream
    try:
        assert fszlib.fsz_set_schedule_ex(dict(decompress_ticket_chunks=ticket, decompress_records=16,
                                               min_tickets_per_cta=0)) == fszlib.OK
        fszlib.fsz_set_test_hooks(0, 20_000_000)
        if batch:
            assert d.run() == fszlib.OK and d.status()[0] == fszlib.ERR_TIMEOUT
        else:
            assert fszlib.fsz_decompress(s.data_ptr(), s.numel(), out.data_ptr(), n, ws.ptr, ws.bytes, sp) == fszlib.OK
            assert fszlib.fsz_check(ws.ptr, sp) == fszlib.ERR_TIMEOUT
    finally:
        fszlib.fsz_set_test_hooks(2 ** 64 - 1, 0)
        fszlib.fsz_set_schedule_ex(None)
    first = ticket * CHUNK
    assert bool((out[:first] == 7.0).all()) and torch.equal(out[first:], want[first:])


@pytest.mark.parametrize("ticket,records", [(4, 16), (4, 9), (3, 7), (2, 4)])
@pytest.mark.parametrize("held", [0, 1])
def test_full_tickets_up_to_the_tail(fszlib, ticket, records, held):
    """Chunk counts around the point where a launch's tickets become smaller, with tickets that are
    held (0) or that may shrink there (1), against the default schedule's reconstruction."""
    dev = _cuda()
    ctas = fszlib.fsz_get_schedule_limits()["sms"]
    for chunks in (ticket * ctas, 16 * ctas, 16 * ctas + ticket + 1, 19 * ctas + 3):
        n = chunks * CHUNK - 77
        s = fszlib.compress(inputs.grf((n,), 7, "cuda"), 1e-3)[0]
        want = fszlib.decompress(s, n=n).clone()
        try:
            assert fszlib.fsz_set_schedule_ex(dict(decompress_ctas_per_sm=1, decompress_ticket_chunks=ticket,
                                                   decompress_records=records,
                                                   min_tickets_per_cta=held)) == fszlib.OK
            got = fszlib.decompress(s, n=n, out=torch.zeros(n, dtype=torch.float32, device=dev))
        finally:
            fszlib.fsz_set_schedule_ex(None)
        assert torch.equal(got, want)
