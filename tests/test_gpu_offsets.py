"""Decompression's byte offsets (sums of chunk sizes read from the rate headers) at the
edges of their 32-chunk blocks and of the tickets, alone, in batches and with two calls
running at once, against the oracle's reconstruction or the serial call's."""
import numpy as np
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHUNK = 8192
# chunks: around one block, two blocks, the ticket sizes 1-4 of a small and a large launch, and
# a field long enough that few CTAs reach the smaller tickets of a launch's end
CHUNKS = [1, 2, 5, 31, 32, 33, 63, 64, 65, 97, 700]


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _field(n, seed):
    """Rates that differ from chunk to chunk, so that no two prefixes are alike."""
    rng = np.random.default_rng(seed)
    scale = np.repeat(10.0 ** rng.uniform(-3, 0, -(-n // 1000)), 1000)[:n]
    return (inputs.sinusoids(n, seed=seed) + scale * rng.standard_normal(n)).astype(np.float32)


@pytest.mark.parametrize("off", [-1, 0, 1])
def test_offsets_at_block_edges(fszlib, oracle, off):
    dev = _cuda()
    xs = [_field(max(1, c * CHUNK + off), c) for c in CHUNKS]
    refs = [oracle.compress(x, 1e-3, oracle.REL) for x in xs]
    want = [oracle.decompress(r).view(np.uint32) for r in refs]
    dev_streams = [torch.from_numpy(np.frombuffer(r, np.uint8).copy()).to(dev) for r in refs]
    scheds = [None, dict(decompress_ticket_chunks=4, decompress_records=8, min_tickets_per_cta=0),
              dict(decompress_ctas_per_sm=1, decompress_ticket_chunks=3, decompress_records=6,
                   min_tickets_per_cta=0),
              dict(decompress_ticket_chunks=1, decompress_records=2, min_tickets_per_cta=0)]
    try:
        for sched in scheds:
            assert fszlib.fsz_set_schedule_ex(sched) == fszlib.OK
            for s, x, w in zip(dev_streams, xs, want):
                y = fszlib.decompress(s, n=x.size).cpu().numpy()
                assert np.array_equal(y.view(np.uint32), w)
            b = fszlib.DecompressBatch(dev_streams, [x.size for x in xs], device=dev)
            assert b.run() == fszlib.OK and b.status()[0] == fszlib.OK
            for i, w in enumerate(want):
                assert np.array_equal(b.output(i).cpu().numpy().view(np.uint32), w)
    finally:
        fszlib.fsz_set_schedule_ex(None)


@pytest.mark.parametrize("ticket,records", [(4, 16), (4, 9), (3, 7), (2, 4), (1, 16)])
def test_tickets_from_the_first_to_the_tail(fszlib, ticket, records):
    """Chunk counts around the point where a launch's tickets become smaller, against the
    default schedule's reconstruction."""
    dev = _cuda()
    ctas = fszlib.fsz_get_schedule_limits()["sms"]     # one CTA per SM
    for chunks in (16 * ctas - 1, 16 * ctas, 16 * ctas + 1, 16 * ctas + ticket + 1, 21 * ctas + 3):
        n = chunks * CHUNK - 77
        x = inputs.grf((n,), 7, "cuda")
        s = fszlib.compress(x, 1e-3, fszlib.EB_REL)[0]
        want = fszlib.decompress(s, n=n).clone()
        try:
            assert fszlib.fsz_set_schedule_ex(dict(decompress_ctas_per_sm=1, decompress_ticket_chunks=ticket,
                                                   decompress_records=records, min_tickets_per_cta=0)) == fszlib.OK
            out = torch.zeros(n, dtype=torch.float32, device=dev)
            got = fszlib.decompress(s, n=n, out=out)
        finally:
            fszlib.fsz_set_schedule_ex(None)
        assert torch.equal(got, want)
        eb = fszlib.fsz_read_header(s[:64].cpu().numpy().tobytes())
        err = (x.reshape(-1).double() - got.double()).abs().max().item()
        assert err <= 1e-3 * (x.max() - x.min()).item() * (1 + 1e-6) and eb["n"] == n


def test_offsets_with_two_calls_at_once(fszlib):
    """Two streams decompress large fields together: CTAs that get an SM late stand far behind
    the tickets already taken, so their next offset spans many blocks."""
    dev = _cuda()
    n = 1 << 26
    xs = [inputs.grf((64, 1024, 1024), seed, "cuda").reshape(-1) for seed in (1, 2)]
    sts = [fszlib.compress(x, 1e-3, fszlib.EB_REL)[0].clone() for x in xs]
    want = [fszlib.decompress(s, n=n).clone() for s in sts]
    lanes = [torch.cuda.Stream(dev) for _ in sts]
    wss = [fszlib.Workspace(n, dev) for _ in sts]
    outs = [torch.empty(n, dtype=torch.float32, device=dev) for _ in sts]
    for rep in range(6):
        for o in outs:
            o.zero_()
        torch.cuda.synchronize()
        for s, lane, ws, o in zip(sts, lanes, wss, outs):
            assert fszlib.fsz_decompress(s.data_ptr(), s.numel(), o.data_ptr(), n, ws.ptr, ws.bytes,
                                         lane.cuda_stream) == fszlib.OK
        torch.cuda.synchronize()
        for w, o, ws, lane in zip(want, outs, wss, lanes):
            assert fszlib.fsz_check(ws.ptr, lane.cuda_stream) == fszlib.OK
            assert torch.equal(o, w)


def test_a_refused_stream_leaves_the_output_alone(fszlib, oracle):
    """A preamble that the set-up refuses: nothing is decoded, whatever the headers say."""
    dev = _cuda()
    x = _field(40 * CHUNK + 5, 3)
    s = np.frombuffer(oracle.compress(x, 1e-3, oracle.REL), np.uint8).copy()
    for at, value, status in ((0, 0, fszlib.ERR_CORRUPT), (13, 0x7F, fszlib.ERR_CORRUPT),
                              (16, 1, fszlib.ERR_CORRUPT), (51, 0xFF, fszlib.ERR_CORRUPT),
                              (53, 1, fszlib.ERR_INVALID_ARG)):
        bad = s.copy()
        bad[at] = value
        sd = torch.from_numpy(bad).to(dev)
        out = torch.full((x.size,), 7.0, dtype=torch.float32, device=dev)
        with pytest.raises(fszlib.FszError) as e:
            fszlib.decompress(sd, n=x.size, out=out)
        assert e.value.status == status
        assert bool((out == 7.0).all())
