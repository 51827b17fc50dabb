"""The value-range pass at the edges of its chunks, segments and CTA ranges: the step in
each stream's preamble against the oracle's, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CHUNK = 8192
SIZES = [1, 2, 3, 4, 5, 7, CHUNK - 1, CHUNK, CHUNK + 1, CHUNK + 3, 2 * CHUNK + 1021, 5 * CHUNK + 4093]


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


def _field(n, where, seed, dev):
    """Values in (-1, 1) with the field's minimum and maximum at its first or last elements."""
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    x = torch.rand(n, generator=g, device=dev) * 2.0 - 1.0
    if where == "first":
        x[0], x[min(1, n - 1)] = -3.0 - seed, 2.0 + seed
    else:
        x[n - 1], x[max(0, n - 2)] = 3.0 + seed, -2.0 - seed
    return x


def _step(oracle, x, rel):
    lo, hi, fin = oracle.stats(x)
    return np.float32(oracle.params(oracle.REL, rel, lo, hi, fin, x.size).s)


def _steps(fszlib, batch):
    assert batch.run() == fszlib.OK
    assert batch.status()[0] == fszlib.OK
    sizes = batch.sizes.cpu().tolist()
    return [np.float32(fszlib.fsz_read_header(batch.stream(i, sizes)[:64].cpu().numpy().tobytes())["step"])
            for i in range(len(batch.n))]


@pytest.mark.parametrize("where", ["first", "last"])
def test_steps_of_many_small_ragged_fields(fszlib, oracle, where):
    dev = _cuda()
    xs = [_field(n, where, k, dev) for k, n in enumerate(SIZES * 7)]  # several fields per CTA range
    got = _steps(fszlib, fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs]))
    assert got == [_step(oracle, x.cpu().numpy(), 1e-3) for x in xs]
    for x, s in zip(xs[:len(SIZES)], got):   # and one call per field
        sb, _ = fszlib.compress(x, 1e-3, fszlib.EB_REL)
        assert np.float32(fszlib.fsz_read_header(sb[:64].cpu().numpy().tobytes())["step"]) == s


def test_steps_when_a_cta_range_spans_several_segments(fszlib, oracle):
    """One CTA per SM and enough chunks that each takes more than one 64-chunk segment."""
    dev = _cuda()
    sms = fszlib.fsz_get_schedule_limits()["sms"]
    big = sms * 70 * CHUNK + 5
    xs = [_field(n, w, k, dev) for k, (n, w) in enumerate([(3, "last"), (big, "last"), (CHUNK + 1, "first"), (9, "last")])]
    try:
        assert fszlib.fsz_set_schedule(1, 0, 0) == fszlib.OK
        got = _steps(fszlib, fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-2) for x in xs]))
    finally:
        fszlib.fsz_set_schedule_ex(None)
    assert got == [_step(oracle, x.cpu().numpy(), 1e-2) for x in xs]


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("n", [1, 5, CHUNK + 3, 2 * CHUNK])
def test_a_non_finite_value_refuses_its_field_only(fszlib, n, bad):
    dev = _cuda()
    for at in {0, n // 2, n - 1}:
        xs = [_field(m, "last", 1, dev) for m in (n, n, 7)]
        xs[1][at] = bad
        b = fszlib.CompressBatch([(x, (x.numel(),), fszlib.EB_REL, 1e-3) for x in xs])
        assert b.run() == fszlib.OK
        assert b.status()[1] == [fszlib.OK, fszlib.ERR_NONFINITE, fszlib.OK]
