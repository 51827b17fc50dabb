"""Calls queued back to back on one stream, each reading what the one before wrote: the
kernels of a call may start under the end of the work before it, and must still see all of
it. Streams and values equal those of the same calls with a wait after each."""
import numpy as np
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("n", [1, 4097, 8192 * 9 + 5, 1 << 20, (1 << 23) + 3])
def test_chained_calls_without_waits(fszlib, n):
    dev = _cuda()
    rounds = 6
    rng = np.random.default_rng(n)
    base = torch.from_numpy(inputs.sinusoids(n, seed=1)).to(dev)
    srcs = [(base * float(s) + float(o)).contiguous()
            for s, o in zip(rng.uniform(0.5, 50.0, rounds), rng.uniform(-9.0, 9.0, rounds))]
    cap, dims = fszlib.fsz_compress_bound(n), fszlib.make_dims((n,))

    def chain(wait):
        x = torch.empty_like(base)
        y = torch.empty(max(n, 4), dtype=torch.float32, device=dev)
        ws = fszlib.Workspace(n, dev)   # one workspace for every call
        sp = torch.cuda.current_stream().cuda_stream
        outs = []
        for src in srcs:
            a = torch.zeros(cap, dtype=torch.uint8, device=dev)
            b = torch.zeros(cap, dtype=torch.uint8, device=dev)
            nb = torch.zeros(2, dtype=torch.int64, device=dev)
            if wait:
                torch.cuda.synchronize()
            x.copy_(src)                               # a kernel writes the input just before
            for inp, eb, out, k in ((x, 1e-3, a, 0), (y, 1e-2, b, 1)):
                assert fszlib.fsz_compress(inp.data_ptr(), dims, fszlib.EB_REL, eb, out.data_ptr(), cap,
                                           nb.data_ptr() + 8 * k, ws.ptr, ws.bytes, sp) == fszlib.OK
                if wait:
                    torch.cuda.synchronize()
                if k == 0:                             # the stream just written, its bound as size
                    assert fszlib.fsz_decompress(a.data_ptr(), cap, y.data_ptr(), y.numel(), ws.ptr,
                                                 ws.bytes, sp) == fszlib.OK
                    if wait:
                        torch.cuda.synchronize()
            outs += [a, b, nb, y[:n].clone()]
        torch.cuda.synchronize()
        return outs

    for got, want in zip(chain(False), chain(True)):
        assert torch.equal(got.view(torch.uint8), want.view(torch.uint8))


def test_graph_of_chained_batches_replays(fszlib):
    """A compression and a decompression of its streams captured into one graph."""
    dev = _cuda()
    sizes = [1, 300, 9000, 70001, 8192 * 40]
    xs = [torch.from_numpy(inputs.sinusoids(m, seed=m % 3)).to(dev) for m in sizes]
    c = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    assert c.run() == fszlib.OK
    slots = [c.arena[c.offsets[i]:c.offsets[i] + c.caps[i]] for i in range(len(xs))]
    d = fszlib.DecompressBatch(slots, sizes, device=dev)
    assert d.run() == fszlib.OK and d.status()[0] == fszlib.OK
    g = torch.cuda.CUDAGraph()
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(g, stream=side):
        assert c.run() == fszlib.OK and d.run() == fszlib.OK
    for scale in (1.0, 7.5):
        for x in xs:
            x.mul_(scale)
        c.arena.zero_()
        d.arena.zero_()
        g.replay()
        torch.cuda.synchronize()
        for i, x in enumerate(xs):
            ref, nb = fszlib.compress(x, 1e-3, fszlib.EB_REL)
            assert int(c.sizes[i]) == nb and torch.equal(c.arena[c.offsets[i]:c.offsets[i] + nb], ref)
            assert torch.equal(d.output(i), fszlib.decompress(ref, n=x.numel()))


@pytest.mark.parametrize("n", [1, 8192 * 3 + 7, 8192 * 700 + 11])
def test_a_refused_field_between_good_ones(fszlib, n):
    """The compression kernel takes its first chunks before the field's step is known: a field
    that then has none writes nothing, and the calls around it are whole."""
    dev = _cuda()
    good = torch.from_numpy(inputs.sinusoids(n, seed=2)).to(dev)
    cap, dims = fszlib.fsz_compress_bound(n), fszlib.make_dims((n,))
    want = fszlib.compress(good, 1e-3)[0].clone()
    ws = fszlib.Workspace(n, dev)
    sp = torch.cuda.current_stream().cuda_stream
    x = good.clone()
    outs = [torch.full((cap,), 0xA5, dtype=torch.uint8, device=dev) for _ in range(3)]
    nb = torch.zeros(3, dtype=torch.int64, device=dev)
    for k, out in enumerate(outs):
        x.copy_(good)
        if k == 1:
            x[n - 1] = float("inf")
        assert fszlib.fsz_compress(x.data_ptr(), dims, fszlib.EB_REL, 1e-3, out.data_ptr(), cap,
                                   nb.data_ptr() + 8 * k, ws.ptr, ws.bytes, sp) == fszlib.OK
        if k == 1:
            assert fszlib.fsz_check(ws.ptr, sp) == fszlib.ERR_NONFINITE
    assert fszlib.fsz_check(ws.ptr, sp) == fszlib.OK
    assert nb.tolist() == [want.numel(), 0, want.numel()]
    for out in (outs[0], outs[2]):
        assert torch.equal(out[:want.numel()], want) and bool((out[want.numel():] == 0xA5).all())
    assert bool((outs[1] == 0xA5).all())


@pytest.mark.parametrize("n", [300, 8192 * 40 + 3])
def test_captured_behind_copies_and_joins(fszlib, n):
    """A captured call whose first kernel follows a copy, a fill, or the join of two streams."""
    dev = _cuda()
    host = [torch.from_numpy(inputs.sinusoids(n, seed=s)).pin_memory() for s in (3, 4)]
    cap, dims = fszlib.fsz_compress_bound(n), fszlib.make_dims((n,))
    x, y = torch.zeros(n, device=dev), torch.zeros(n, device=dev)
    back = torch.zeros(max(n, 4), device=dev)
    a, b = (torch.zeros(cap, dtype=torch.uint8, device=dev) for _ in range(2))
    nb = torch.zeros(2, dtype=torch.int64, device=dev)
    wa, wb = fszlib.Workspace(n, dev), fszlib.Workspace(n, dev)
    feed = host[0].clone().pin_memory()
    fszlib.compress(host[0].to(dev), 1e-3)              # (launch settings, before the capture)
    fszlib.decompress(fszlib.compress(host[0].to(dev), 1e-3)[0], n=n)

    def comp(src, out, k, ws):
        sp = torch.cuda.current_stream().cuda_stream
        return fszlib.fsz_compress(src.data_ptr(), dims, fszlib.EB_REL, 1e-3, out.data_ptr(), cap,
                                   nb.data_ptr() + 8 * k, ws.ptr, ws.bytes, sp)

    g = torch.cuda.CUDAGraph()
    main, side = torch.cuda.Stream(dev), torch.cuda.Stream(dev)
    with torch.cuda.graph(g, stream=main):
        x.copy_(feed, non_blocking=True)
        assert comp(x, a, 0, wa) == fszlib.OK           # behind a copy
        side.wait_stream(main)
        with torch.cuda.stream(side):
            y.copy_(x)
            y.mul_(3.0)
        back.zero_()
        main.wait_stream(side)
        assert comp(y, b, 1, wb) == fszlib.OK           # behind a fill and another stream
        assert fszlib.fsz_decompress(b.data_ptr(), cap, back.data_ptr(), back.numel(), wa.ptr, wa.bytes,
                                     main.cuda_stream) == fszlib.OK
    for h in host:
        feed.copy_(h)
        g.replay()
        torch.cuda.synchronize()
        for src, out, k in ((h.to(dev), a, 0), (h.to(dev) * 3.0, b, 1)):
            ref, m = fszlib.compress(src, 1e-3)
            assert int(nb[k]) == m and torch.equal(out[:m], ref[:m])
        assert torch.equal(back[:n], fszlib.decompress(b[:int(nb[1])].clone(), n=n))
