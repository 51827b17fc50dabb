"""Compression of batches on both sides of the 64 fields up to which the value-range kernel plans for
itself, with refused descriptors among them, and of so few and long fields that a CTA's range takes
several segments: statuses, sizes and streams are the one-field call's."""
import ctypes

import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("nfields", [1, 31, 32, 33, 63, 64, 65])
def test_refused_descriptors_among_good_ones(fszlib, nfields):
    dev = _cuda()
    src = torch.from_numpy(inputs.sinusoids(1 << 20, seed=4)).to(dev)
    sizes = [(8192, 1, 70000, 0, 8193, 500000, 255)[k % 7] for k in range(nfields)]
    xs = [src[64 * k:64 * k + n].clone() for k, n in enumerate(sizes)]
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    arr = (fszlib.FszCField * nfields).from_buffer_copy(b.table.cpu().numpy().tobytes())
    want = [fszlib.OK] * nfields
    for k in range(nfields):
        f = arr[k]
        if k % 8 == 2:
            f.eb, want[k] = -1.0, fszlib.ERR_INVALID_ARG
        elif k % 8 == 4 and sizes[k]:
            f.in_, want[k] = f.in_ + 4, fszlib.ERR_ALIGN
        elif k % 8 == 5:
            f.out_capacity, want[k] = 40, fszlib.ERR_CAPACITY
        elif k % 8 == 6:
            f.dims.ndim, want[k] = 7, fszlib.ERR_INVALID_ARG
        elif k % 8 == 7 and sizes[k]:
            xs[k][sizes[k] - 1], want[k] = float("inf"), fszlib.ERR_NONFINITE
    b.table.copy_(torch.frombuffer(bytearray(bytes(arr)), dtype=torch.uint8))
    b.ws.fill_(0xFF)
    for _ in range(2):                     # the second call over the first one's workspace
        b.sizes.zero_()
        b.arena.fill_(0xA5)
        assert b.run() == fszlib.OK
        status, per = b.status()
        assert per == want
        assert (status == fszlib.OK) == all(w == fszlib.OK for w in want)
        ks = b.sizes.cpu().tolist()
        for k in range(nfields):
            if want[k] == fszlib.OK:
                ref, nb = fszlib.compress(xs[k], 1e-3)
                assert ks[k] == nb and torch.equal(b.stream(k, ks), ref), k
            else:
                assert ks[k] == 0, k


def test_more_chunks_than_the_workspace_holds(fszlib):
    dev = _cuda()
    xs = [torch.from_numpy(inputs.sinusoids(1 << 18, seed=s)).to(dev) for s in (1, 2, 3)]
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    b.arena.zero_()
    sp = torch.cuda.current_stream().cuda_stream
    few = fszlib.fsz_batch_workspace_bytes(8192, 3)
    assert fszlib.fsz_compress_batched(b.table.data_ptr(), 3, 8192, b.ws.data_ptr(), few, sp) == fszlib.OK
    assert fszlib.fsz_check(b.ws.data_ptr(), sp) == fszlib.ERR_WORKSPACE
    assert int(torch.count_nonzero(b.arena)) == 0 and b.sizes.tolist() == [0, 0, 0]


def test_ranges_of_several_segments(fszlib):
    """2^29 values: 86 chunks per CTA, more than a segment's 64, the fields' border inside one."""
    dev = _cuda()
    g = torch.Generator(device=dev).manual_seed(8)
    sizes = [(1 << 28) + 8192 * 5 + 3, (1 << 28) - 8192 * 9 + 1]
    xs = [torch.randn(n, device=dev, generator=g) for n in sizes]
    xs[0][sizes[0] - 2] = 40.0             # each field's extremes near its ends
    xs[1][1], xs[1][sizes[1] - 1] = -55.0, 60.0
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    assert b.run() == fszlib.OK and b.status() == (fszlib.OK, [fszlib.OK] * 2)
    ks = b.sizes.cpu().tolist()
    for k, x in enumerate(xs):
        ref, nb = fszlib.compress(x, 1e-3)
        assert ks[k] == nb and torch.equal(b.stream(k, ks), ref)


@pytest.mark.parametrize("nfields", [3, 64, 65, 200])
def test_fields_refused_in_one_call_and_not_in_the_next(fszlib, nfields):
    """Queued without waits: the compression kernel takes its first chunks before their fields' steps
    are known."""
    dev = _cuda()
    good = [torch.from_numpy(inputs.sinusoids(20000 + 7 * k, seed=k % 5)).to(dev) for k in range(nfields)]
    xs = [x.clone() for x in good]
    b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs], device=dev)
    sizes, arenas, statuses = [], [], []
    torch.cuda.synchronize()
    for call in range(4):
        for k in range(nfields):
            xs[k].copy_(good[k])
            if (k + call) % 3 == 0:
                xs[k][11 * call + k] = float("nan")
        b.arena.fill_(0xA5)
        b.sizes.zero_()
        assert b.run() == fszlib.OK
        sizes.append(b.sizes.clone())
        arenas.append(b.arena.clone())
        if call == 3:
            statuses = b.status()[1]
    refs = [fszlib.compress(x, 1e-3)[0] for x in good]
    for call in range(4):
        ks = sizes[call].tolist()
        for k in range(nfields):
            slot = arenas[call][b.offsets[k]:b.offsets[k] + b.caps[k]]
            if (k + call) % 3 == 0:
                assert ks[k] == 0
            else:
                assert ks[k] == refs[k].numel() and torch.equal(slot[:ks[k]], refs[k]), (call, k)
    assert statuses == [fszlib.ERR_NONFINITE if (k + 3) % 3 == 0 else fszlib.OK for k in range(nfields)]
