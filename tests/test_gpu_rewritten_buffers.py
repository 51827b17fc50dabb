"""Descriptors, fields and streams rewritten in place between batched calls that are queued without
waits: the kernels of a call read them before their predecessor has ended, and must see what was
written last. Every preamble, rate header and descriptor differs from one call to the next."""
import numpy as np
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CALLS, MOST = 6, 30000


def _write(how, dst, src, pinned):
    if how == "kernel":
        torch.bitwise_or(src, 0, out=dst)
    elif how == "copy":
        dst.copy_(src)
    else:
        dst.copy_(pinned, non_blocking=True)


# up to 64 fields are planned by the value-range kernel and up to 512 by the sizing kernel for itself
@pytest.mark.parametrize("how", ["kernel", "copy", "host"])
@pytest.mark.parametrize("nfields", [5, 70, 520])
def test_everything_rewritten_between_calls(fszlib, nfields, how):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(nfields)
    base = torch.from_numpy(inputs.sinusoids(1 << 18, seed=6)).to(dev)
    noise = torch.from_numpy(rng.standard_normal(1 << 18).astype(np.float32)).to(dev)
    buf = torch.zeros(nfields * MOST, dtype=torch.float32, device=dev)
    slots = [buf[k * MOST:(k + 1) * MOST] for k in range(nfields)]
    c = fszlib.CompressBatch([(s, (MOST,), fszlib.EB_REL, 1e-3) for s in slots], device=dev)
    streams = torch.zeros_like(c.arena)
    d = fszlib.DecompressBatch([streams[c.offsets[k]:c.offsets[k] + c.caps[k]] for k in range(nfields)],
                               [MOST] * nfields, device=dev)
    ctable = (fszlib.FszCField * nfields).from_buffer_copy(c.table.cpu().numpy().tobytes())
    dtable = (fszlib.FszDField * nfields).from_buffer_copy(d.table.cpu().numpy().tobytes())
    calls = []
    for i in range(CALLS):                 # call i's fields, descriptors and streams, made beforehand
        sizes = rng.integers(1, MOST + 1, nfields)
        order = rng.permutation(nfields)
        values = torch.zeros_like(buf)
        ct = (fszlib.FszCField * nfields)()
        dt = (fszlib.FszDField * nfields)()
        refs, outs, packed = [], [], torch.zeros_like(streams)
        for k in range(nfields):           # descriptor k: slot order[k], sizes[k] values
            s, n = int(order[k]), int(sizes[k])
            at = 64 * int(rng.integers(0, 3000))
            x = base[at:at + n] * 4 + noise[at:at + n] * float(10.0 ** rng.uniform(-3, 0))
            values[s * MOST:s * MOST + n] = x
            ct[k], dt[k] = ctable[s], dtable[s]
            ct[k].dims = fszlib.make_dims((n,))
            ct[k].eb = float(10.0 ** rng.uniform(-4, -2))
            ct[k].out_bytes = ctable[k].out_bytes
            ref, nb = fszlib.compress(x.contiguous(), ct[k].eb)
            refs.append(ref.clone())
            outs.append(fszlib.decompress(ref, n=n).clone())
            packed[c.offsets[s]:c.offsets[s] + nb] = ref
        tabs = [torch.frombuffer(bytearray(bytes(t)), dtype=torch.uint8) for t in (ct, dt)]
        sets = [(buf.view(torch.uint8), values.view(torch.uint8)), (streams, packed),
                (c.table, tabs[0].to(dev)), (d.table, tabs[1].to(dev))]
        calls.append((order, sizes, refs, outs, [(t, v, v.cpu().pin_memory()) for t, v in sets]))
    torch.cuda.synchronize()
    got = []
    for order, sizes, refs, outs, sets in calls:
        for dst, src, pinned in sets:
            _write(how, dst, src, pinned)
        assert c.run() == fszlib.OK and d.run() == fszlib.OK
        got.append((c.arena.clone(), c.sizes.clone(), d.arena.clone()))
    torch.cuda.synchronize()
    for (order, sizes, refs, outs, _), (arena, nbytes, values) in zip(calls, got):
        nbytes = nbytes.tolist()
        for k in range(nfields):
            s = int(order[k])
            assert nbytes[k] == refs[k].numel(), k
            assert torch.equal(arena[c.offsets[s]:c.offsets[s] + nbytes[k]], refs[k]), k
            assert torch.equal(values[d.offsets[s]:d.offsets[s] + int(sizes[k])], outs[k]), k
