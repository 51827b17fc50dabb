"""The work that a user of this library has it do, as cases that can be timed and compared.

A case is one call of a public entry point on data of the kind and size that the library's
own workloads have (``paper_2607_15413_gb300.inputs``): served requests of 16 KiB to
256 MiB, the 2^20-sample signal, 512^3 simulation fields, particle arrays, and batches of
many fields of mixed size. ``prepare`` makes what a program holds before the call, ``run``
makes the call, ``work`` counts the bytes and operations it cannot do without, and
``exact`` restates the reconstruction in float64 with plain torch.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2607_15413_gb300 import fsz, inputs

# Stream bits per value of each class at REL 1e-2, 1e-3 and 1e-4 (for the output bytes of
# `work`; the streams' sizes depend on the data).
_BITS = {"signal": (2.5, 4.0, 7.0), "smooth": (4.4, 7.7, 11.0),
         "particle": (3.4, 5.5, 8.3), "zero_heavy": (0.7, 2.4, 4.5)}

# The three source fields that requests of a batch are cut from.
_POOL_SHAPE = (64, 512, 512)


def listed():
    return [
        # The smallest served request, through the Python call that checks the status and
        # returns the stream or the values: all latency.
        dict(name="compress_16k_call", kind="compress", entry="call", cls="signal", shape="4096",
             mode="rel", eb=1e-3),
        dict(name="decompress_16k_call", kind="decompress", entry="call", cls="signal", shape="4096",
             mode="rel", eb=1e-3),
        # The 2^20-sample signal with buffers that the program keeps: one call among many on
        # a stream, launches and the start and end of each kernel count.
        dict(name="compress_signal_4m", kind="compress", entry="kept", cls="signal", shape="1048576",
             mode="rel", eb=1e-3),
        dict(name="decompress_signal_4m", kind="decompress", entry="kept", cls="signal",
             shape="1048576", mode="rel", eb=1e-3),
        # An ordinary simulation field with a large offset and zero regions, odd extents and a
        # ragged last tile, under an absolute bound.
        dict(name="compress_slabs_31m_abs", kind="compress", entry="kept", cls="zero_heavy",
             shape="121,251,269", mode="abs", eb=0.05),
        # An ordinary particle array of odd length at a tight bound.
        dict(name="decompress_particles_61m", kind="decompress", entry="kept", cls="particle",
             shape="16000003", mode="rel", eb=1e-4),
        # The headline: a 512^3 field at REL 1e-3, each direction.
        dict(name="compress_grf_512cubed", kind="compress", entry="kept", cls="smooth",
             shape="512,512,512", mode="rel", eb=1e-3),
        dict(name="decompress_grf_512cubed", kind="decompress", entry="kept", cls="smooth",
             shape="512,512,512", mode="rel", eb=1e-3),
        # A batch of 32 requests (what the server launches at a time), log-uniform sizes, mixed
        # classes and bounds, as one batched call over a field table.
        dict(name="compress_batch_32", kind="compress_batch", fields=32, lo=4096, hi=1 << 24, mix=5),
        dict(name="decompress_batch_32", kind="decompress_batch", fields=32, lo=4096, hi=1 << 24, mix=5),
        # A tile configuration other than the default (64-element blocks), each direction.
        dict(name="compress_tiles_64x8", kind="compress_tiled", cls="smooth", shape="256,256,256",
             mode="rel", eb=1e-3, block=64, blocks=8),
        dict(name="decompress_tiles_64x8", kind="decompress_tiled", cls="smooth", shape="256,256,256",
             mode="rel", eb=1e-3, block=64, blocks=8),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))

    kind = rng.choice(["compress", "decompress", "compress", "decompress", "compress_batch",
                       "decompress_batch", "compress_tiled", "decompress_tiled"])
    if kind.endswith("batch"):
        return dict(kind=kind, fields=rng.randrange(3, 65), lo=4096, hi=log_int(1 << 16, 1 << 22),
                    mix=rng.randrange(1 << 20))
    cls = rng.choice(["signal", "smooth", "particle", "zero_heavy"])
    # (the signal is made on the host, so its sizes end at 2^22)
    n = log_int(4096, (1 << 22) if cls == "signal" else (1 << 25) if kind.endswith("tiled") else (1 << 26))
    ndim = 1 if cls in ("signal", "particle") else rng.choice([2, 3])
    if ndim == 1:
        shape = (n,)
    elif ndim == 2:
        a = max(3, int(math.sqrt(n) * rng.uniform(0.6, 1.4)))
        shape = (a, max(3, n // a))
    else:
        a = max(3, int(n ** (1 / 3) * rng.uniform(0.6, 1.4)))
        b = max(3, int(math.sqrt(n / a)))
        shape = (a, b, max(3, n // (a * b)))
    mode = rng.choice(["rel", "rel", "abs"])
    eb = rng.choice([1e-2, 1e-3, 1e-4])
    if mode == "abs":  # of each class's usual range (about 6, 9, 2700 and 290)
        eb *= {"signal": 6.0, "smooth": 9.0, "particle": 2700.0, "zero_heavy": 290.0}[cls]
    case = dict(kind=kind, cls=cls, shape=",".join(str(s) for s in shape), mode=mode, eb=eb)
    if kind.endswith("tiled"):
        case["block"], case["blocks"] = rng.choice(fsz.TILE_CONFIGS)
    else:
        case["entry"] = rng.choice(["call", "kept", "kept"])
    return case


# ------------------------------------------------------------------ inputs

def _shape(case):
    return tuple(int(s) for s in case["shape"].split(","))


def _field(case, seed):
    """The case's field on the GPU, in its shape."""
    shape, seed = _shape(case), seed % (1 << 31)
    n = math.prod(shape)
    if case["cls"] == "signal":
        return torch.from_numpy(inputs.sinusoids(n, seed)).to("cuda").reshape(shape)
    if case["cls"] == "smooth":
        return inputs.grf(shape, seed, "cuda")
    if case["cls"] == "particle":
        return inputs.particles(n, seed, "cuda", ncenters=max(16, n // 2048)).reshape(shape)
    return inputs.zero_slabs(shape, seed, "cuda").contiguous()


def _mode(case):
    return fsz.EB_ABS if case["mode"] == "abs" else fsz.EB_REL


def _requests(case):
    """The batch's requests: (source, element offset's fraction, elements, REL), by the case alone."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["fields"]):
        n = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))
        out.append((rng.randrange(3), rng.random(), n, rng.choice([1e-2, 1e-3, 1e-4])))
    return out


def _batch_fields(case, seed):
    """The batch's fields: windows at 16-byte boundaries of a smooth, a particle-like and a
    zero-heavy source."""
    seed = seed % (1 << 31)
    g = inputs.grf(_POOL_SHAPE, seed, "cuda")
    pool = [g.reshape(-1), inputs.particles(g.numel(), seed, "cuda"),
            inputs.zero_slabs(_POOL_SHAPE, seed, "cuda", base=g).reshape(-1)]
    fields = []
    for k, at, n, rel in _requests(case):
        off = int(at * (pool[k].numel() - n)) // 4 * 4
        fields.append((pool[k][off:off + n].clone(), (n,), fsz.EB_REL, rel))
    return fields


def prepare(case, seed):
    """What a program holds before the call: its field or stream, and the buffers, workspace
    or batch that it keeps. Buffers start as zeros, so that their unused ends are equal."""
    kind = case["kind"]
    if kind == "compress_batch":
        batch = fsz.CompressBatch(_batch_fields(case, seed))
        batch.arena.zero_()
        return dict(kind=kind, batch=batch)
    if kind == "decompress_batch":
        fields = _batch_fields(case, seed)
        comp = fsz.CompressBatch(fields)
        fsz._check(comp.run(), "fsz_compress_batched")
        sizes = comp.sizes.cpu().tolist()
        batch = fsz.DecompressBatch([comp.stream(i, sizes).clone() for i in range(len(fields))],
                                    [x.numel() for x, *_ in fields])
        batch.arena.zero_()
        return dict(kind=kind, batch=batch,
                    outs=[batch.output(i) for i in range(len(fields))])
    x = _field(case, seed)
    n = x.numel()
    state = dict(kind=kind, entry=case.get("entry", "call"), n=n, mode=_mode(case), eb=case["eb"])
    if kind.endswith("tiled"):
        ws_bytes = fsz.lib().fsz_tiled_workspace_bytes(n)
        state.update(ws=torch.empty(ws_bytes, dtype=torch.uint8, device="cuda"), ws_bytes=ws_bytes)
    if kind == "compress_tiled":
        cap = fsz.lib().fsz_compress_bound_tiled(n, case["block"], case["blocks"])
        state.update(x=x, block=case["block"], blocks=case["blocks"], dims=fsz.make_dims(x.shape),
                     out=torch.zeros(cap, dtype=torch.uint8, device="cuda"),
                     nbytes=torch.zeros(1, dtype=torch.int64, device="cuda"))
    elif kind == "decompress_tiled":
        state["stream"] = fsz.compress_tiled(x, case["eb"], _mode(case), block=case["block"],
                                             tile_blocks=case["blocks"])[0].clone()
        state["out"] = torch.zeros(n, dtype=torch.float32, device="cuda")
    elif kind == "compress":
        state.update(x=x, dims=fsz.make_dims(x.shape), ws=fsz.Workspace(n),
                     out=torch.zeros(fsz.fsz_compress_bound(n), dtype=torch.uint8, device="cuda"),
                     nbytes=torch.zeros(1, dtype=torch.int64, device="cuda"))
    else:
        state["stream"] = fsz.compress(x, case["eb"], _mode(case))[0].clone()
        if state["entry"] == "kept":
            state.update(ws=fsz.Workspace(n), out=torch.zeros(n, dtype=torch.float32, device="cuda"))
    return state


# ------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "compress_batch":
        batch = state["batch"]
        fsz._check(batch.run(), "fsz_compress_batched")
        return [batch.arena, batch.sizes]
    if kind == "decompress_batch":
        fsz._check(state["batch"].run(), "fsz_decompress_batched")
        return state["outs"]
    sp = torch.cuda.current_stream().cuda_stream
    ws, out = state.get("ws"), state.get("out")
    if kind == "compress_tiled":
        fsz._check(fsz.lib().fsz_compress_tiled(
            state["x"].data_ptr(), state["dims"], state["mode"], state["eb"], state["block"],
            state["blocks"], 0, out.data_ptr(), out.numel(), state["nbytes"].data_ptr(),
            ws.data_ptr(), state["ws_bytes"], sp), "fsz_compress_tiled")
        return [out, state["nbytes"]]
    if kind == "decompress_tiled":
        stream = state["stream"]
        fsz._check(fsz.lib().fsz_decompress_tiled(
            stream.data_ptr(), stream.numel(), out.data_ptr(), out.numel(), ws.data_ptr(),
            state["ws_bytes"], sp), "fsz_decompress_tiled")
        return [out]
    if state["entry"] == "call":
        if kind == "compress":
            _, size = fsz.compress(state["x"], state["eb"], state["mode"], ws=ws, out=out)
            return [out, size]  # (the stream is the buffer's first `size` bytes)
        return [fsz.decompress(state["stream"], n=state["n"])]
    if kind == "compress":
        fsz._check(fsz.fsz_compress(state["x"].data_ptr(), state["dims"], state["mode"], state["eb"],
                                    out.data_ptr(), out.numel(), state["nbytes"].data_ptr(), ws.ptr,
                                    ws.bytes, sp), "fsz_compress")
        return [out, state["nbytes"]]
    stream = state["stream"]
    fsz._check(fsz.fsz_decompress(stream.data_ptr(), stream.numel(), out.data_ptr(), out.numel(),
                                  ws.ptr, ws.bytes, sp), "fsz_decompress")
    return [out]


# ------------------------------------------------------------------ what it cannot do without

def _stream_bytes(n, cls, rel):
    k = 0 if rel > 3e-3 else 1 if rel > 3e-4 else 2
    return n * _BITS[cls][k] / 8


def work(case):
    """4 bytes per value on one side and the stream (its size estimated from the class and
    the bound) on the other; per value, compression multiplies and rounds to quantize and adds
    to the tile's mean, decompression multiplies by the step."""
    if case["kind"].endswith("batch"):
        classes = ("smooth", "particle", "zero_heavy")
        reqs = _requests(case)
        n = sum(r[2] for r in reqs)
        out = sum(_stream_bytes(r[2], classes[r[0]], r[3]) for r in reqs)
    else:
        n = math.prod(_shape(case))
        rel = case["eb"]
        if case["mode"] == "abs":
            rel /= {"signal": 6.0, "smooth": 9.0, "particle": 2700.0, "zero_heavy": 290.0}[case["cls"]]
        out = _stream_bytes(n, case["cls"], rel)
    per = 3 if case["kind"].startswith("compress") else 1
    return {"bytes": int(4 * n + out), "flops": per * n}


# ------------------------------------------------------------------ the values in float64

def _reconstruct(x, mode, eb):
    """The reconstruction of x in float64: the nearest multiple of the step 2e (the
    quantizer's own float32 product, ties to even), e = eb (1 - (3Q + 4) 2^-23) rounded toward
    zero, with eb relative to the value range under "rel" and Q the bound on |q|."""
    lo, hi = float(x.min()), float(x.max())
    top = max(abs(lo), abs(hi))
    if mode == fsz.EB_REL:
        eb = eb * (hi - lo) if hi > lo else (eb * abs(hi) if hi else eb)
    for cap, qmax in ((2.0 ** -4, 174761), (2.0 ** -1, 1398100)):
        q = math.ceil(top / (2.0 * eb * (1.0 - cap))) + 1
        if q <= qmax:
            break
    exact_e = eb * (1.0 - (3 * q + 4) * 2.0 ** -23)
    e = np.float32(exact_e)
    if float(e) > exact_e:
        e = np.nextafter(e, np.float32(0))
    s = np.float32(2) * e
    r = np.float32(1) / s
    return torch.round(x.reshape(-1) * float(r)).double() * float(s)


def exact(case, seed):
    """Streams are bytes and have no such value; reconstructions do."""
    kind = case["kind"]
    if kind.startswith("compress"):
        return None
    if kind == "decompress_batch":
        return [_reconstruct(x, mode, eb) for x, _, mode, eb in _batch_fields(case, seed)]
    return [_reconstruct(_field(case, seed), _mode(case), case["eb"])]
