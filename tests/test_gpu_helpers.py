"""The Python helpers' stream sizes (a pinned host word): every helper, with and without the
status check, on another stream, from several threads, and after a refused call."""
import threading

import numpy as np
import pytest

from paper_2607_15413_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch.device("cuda:0")


@pytest.mark.parametrize("n", [1, 4096, 8192 * 5 + 3])
def test_sizes_of_every_helper(fszlib, oracle, n):
    dev = _cuda()
    x = inputs.sinusoids(n, seed=n % 7)
    xd = torch.from_numpy(x).to(dev)
    ref = oracle.compress(x, 1e-3, oracle.REL)
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream())
    for kw in ({}, {"check": False}, {"stream": side}, {"stream": side, "check": False}):
        for call in (lambda: fszlib.compress(xd, 1e-3, **kw),
                     lambda: fszlib.compress_multipass(xd, 1e-3, **kw)[:2],
                     lambda: fszlib.compress_tiled(xd, 1e-3, **kw)):
            sb, nb = call()
            assert isinstance(nb, int) and nb == len(ref) == sb.numel()
            assert sb.cpu().numpy().tobytes() == ref


def test_sizes_from_several_threads(fszlib, oracle):
    dev = _cuda()
    xs = [inputs.sinusoids(3000 + 517 * k, seed=k) for k in range(8)]
    refs = [oracle.compress(x, 1e-3, oracle.REL) for x in xs]
    bad = []

    def work(k):
        xd = torch.from_numpy(xs[k]).to(dev)
        st = torch.cuda.Stream(dev)
        st.wait_stream(torch.cuda.current_stream())
        for _ in range(30):
            sb, nb = fszlib.compress(xd, 1e-3, stream=st)
            with torch.cuda.stream(st):
                got = sb.cpu().numpy().tobytes()
            if nb != len(refs[k]) or got != refs[k]:
                bad.append(k)

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(xs))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


def test_size_after_a_refusal(fszlib):
    dev = _cuda()
    x = torch.ones(5000, device=dev)
    x[17] = float("nan")
    with pytest.raises(fszlib.FszError) as e:
        fszlib.compress(x, 1e-3)
    assert e.value.status == fszlib.ERR_NONFINITE
    assert fszlib.compress(x, 1e-3, check=False)[1] == 0
    x[17] = 1.0
    assert fszlib.compress(x, 1e-3)[1] > 64
