"""Performance cases: what users of this library have it do, through its
public entry points, over the range of sizes it is used at.

Each case is a dict of plain values.  ``listed()`` gives the fixed ones,
``draw(rng)`` others of the same ranges; ``prepare`` makes what a program holds
before the call (generator, batch or server objects and output memory), ``run``
is one pass, ``work`` the bytes and 64-bit integer operations one pass cannot
do without, and ``exact`` the same outputs from a few lines of torch.

Kinds:
  device    ``Generator.generate`` into device memory the caller owns (``fresh``:
            the program starts its streams over on each pass; else every pass
            continues where the last one stopped)
  call      the same with the output allocated by the call
  checksum  ``Generator.generate_checksum``
  resume    ``Generator.skip`` and then some rows: resuming, or one worker's
            part of a run that is split by iterations
  batch     ``Batch.run`` of many uneven generators
  noalloc   ``rng_batch_generate_noalloc`` of many uneven generators
  serve     a burst of requests to ``Server``, until all results are there
  host      ``Generator.generate_to_host`` into page-locked host memory
"""
import ctypes

import torch

import paper_1609_01257_gb300 as rng
import workloads

_M64 = (1 << 64) - 1
_MB = 1 << 20


def listed():
    return [
        # The smallest call: a few rows of a small generator, as a program that
        # draws numbers as it goes asks for them.  Odd stream count.
        dict(name="call 1000x8", kind="call", streams=1000, rows=8, mode=0),
        # The paper's example size, started over from its hash on every pass.
        dict(name="plain 65536x100", kind="device", streams=1 << 16, rows=100, mode=0, fresh=True),
        # The paper-shaped streaming run, kept on the device: 32 GiB.
        dict(name="stream 4Mx1024", kind="device", streams=1 << 22, rows=1024, mode=0, fresh=True),
        # A stream count off every alignment, the stronger output, continuing.
        dict(name="ragged 1000003x128", kind="device", streams=1_000_003, rows=128, mode=1, fresh=False),
        # Few streams, long sequences.
        dict(name="long 4096x65536", kind="device", streams=4096, rows=65536, mode=0, fresh=True),
        # Very many streams, a few numbers each per call (a Monte Carlo step).
        dict(name="wide 64Mx4", kind="device", streams=1 << 26, rows=4, mode=0, fresh=False),
        # Generate-and-checksum over the streaming run: verification, and the
        # generator's speed without its output.
        dict(name="checksum 4Mx1024", kind="checksum", streams=1 << 22, rows=1024, mode=0),
        # Resuming 16 M streams a long way on.
        dict(name="resume 16M+4", kind="resume", streams=1 << 24, rows=4, mode=0, skip=(1 << 40) + 12345),
        # The batched form at its own workload's size: 512 uneven generators, 8 GiB.
        dict(name="batch 512", kind="batch", count=512, max_streams=1 << 20, max_rows=4096, cap_mb=8192),
        # The allocation-free form as a framework calls it: 64 uneven tensors.
        dict(name="noalloc 64", kind="noalloc", count=64, max_streams=1 << 20, max_rows=64, cap_mb=1024),
        # A burst of requests of the served workload's sizes.
        dict(name="serve 24", kind="serve", count=24, max_streams=1 << 22, max_rows=512, cap_mb=6144),
        # Host-streamed output: 1 GiB over the host link.
        dict(name="host 4Mx32", kind="host", streams=1 << 22, rows=32, mode=0),
    ]


def _log_int(r, lo, hi):
    return max(lo, min(hi, int(lo * (hi / lo) ** r.random())))


def _some(r, lo, hi):
    """A stream count: half of them odd sizes, half multiples of 256."""
    n = _log_int(r, lo, hi)
    return n | 1 if r.random() < 0.5 else max(256, n // 256 * 256)


def draw(rng_):
    r = rng_
    kind = r.choice(["call", "device", "device", "device", "checksum", "resume", "batch", "noalloc", "serve", "host"])
    if kind == "call":
        return dict(kind=kind, streams=_some(r, 256, 1 << 16), rows=_log_int(r, 1, 64), mode=r.choice([0, 1]))
    if kind == "device":
        n = _some(r, 1 << 12, 1 << 26)
        return dict(kind=kind, streams=n, rows=_log_int(r, 1, max(1, (4096 * _MB) // (8 * n))), mode=r.choice([0, 0, 1]),
                    fresh=r.random() < 0.5)
    if kind == "checksum":
        n = _some(r, 1 << 12, 1 << 24)
        return dict(kind=kind, streams=n, rows=_log_int(r, 16, min(65536, max(16, (1 << 31) // n))), mode=r.choice([0, 1]))
    if kind == "resume":
        return dict(kind=kind, streams=_some(r, 1 << 14, 1 << 25), rows=_log_int(r, 1, 16), mode=0, skip=r.getrandbits(48) | 1)
    if kind == "batch":
        return dict(kind=kind, count=_log_int(r, 8, 512), max_streams=_log_int(r, 1 << 14, 1 << 22),
                    max_rows=_log_int(r, 64, 4096), cap_mb=_log_int(r, 256, 4096))
    if kind == "noalloc":
        return dict(kind=kind, count=_log_int(r, 4, 512), max_streams=_log_int(r, 1 << 12, 1 << 20),
                    max_rows=_log_int(r, 8, 256), cap_mb=_log_int(r, 64, 2048))
    if kind == "serve":
        return dict(kind=kind, count=_log_int(r, 4, 48), max_streams=_log_int(r, 1 << 16, 1 << 22),
                    max_rows=_log_int(r, 32, 512), cap_mb=_log_int(r, 512, 6144))
    n = _some(r, 1 << 16, 1 << 22)
    return dict(kind=kind, streams=n, rows=_log_int(r, 1, max(1, (512 * _MB) // (8 * n))), mode=0)


def _instances(case, seed):
    """Uneven sizes by the batched workload's draw rule; the sizes depend on
    the case alone, the run seeds on `seed`."""
    return workloads.batched_instances(
        case["count"], seed_start=seed + 7, size_start=case["count"] + 1007, streams_lo=256,
        streams_hi=case["max_streams"], iters_lo=1, iters_hi=case["max_rows"], cap_bytes=case["cap_mb"] * _MB)


def _offsets(insts):
    """Start of each output in one buffer, on 256-byte boundaries, and its size in values."""
    offs, o = [], 0
    for i in insts:
        offs.append(o)
        o += -(-i.streams * i.iterations // 32) * 32
    return offs, o


class _DeviceMemory:
    """Device memory of the server's, by address, as torch takes it."""

    def __init__(self, addr, values):
        self.__cuda_array_interface__ = {"data": (addr, False), "shape": (values,), "typestr": "<i8", "version": 3}


def prepare(case, seed):
    kind = case["kind"]
    dev = torch.device("cuda")
    s = dict(case=case, kind=kind)
    if kind in ("call", "device", "checksum", "resume", "host"):
        n, t = case["streams"], case["rows"]
        s["gen"] = rng.Generator(n, seed, output_mode=case["mode"])
        if kind == "device" and not case["fresh"]:
            s["gen"].skip(1)  # the states are in memory, as after an earlier call
        if kind in ("device", "resume"):
            s["out"] = torch.empty((t, n), dtype=torch.uint64, device=dev)
        elif kind == "host":
            s["out"] = torch.zeros((t, n), dtype=torch.int64).pin_memory()
        return s
    insts = _instances(case, seed)
    if kind == "serve":
        s["server"] = rng.Server(hbm_budget_bytes=8192 * _MB)
        s["requests"] = [(i.seed, i.streams, i.iterations) for i in insts]
        s["held"], s["views"] = [], {}
        return s
    offs, total = _offsets(insts)
    s["flat"] = torch.zeros(total, dtype=torch.int64, device=dev)
    outs = [s["flat"][o:o + i.streams * i.iterations].view(i.iterations, i.streams) for o, i in zip(offs, insts)]
    lists = [i.streams for i in insts], [i.iterations for i in insts], [i.seed for i in insts]
    if kind == "batch":
        s["batch"] = rng.Batch(*lists, outputs=outs)
    else:
        u64s = ctypes.c_uint64 * len(insts)
        s["lib"] = rng.load()
        s["args"] = [u64s(*v) for v in lists] + [(ctypes.c_void_p * len(insts))(*[o.data_ptr() for o in outs])]
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "call":
        return s["gen"].generate(case["rows"]).view(torch.int64)
    if kind == "device":
        if case["fresh"]:
            s["gen"].init()
        return s["gen"].generate(case["rows"], out=s["out"]).view(torch.int64)
    if kind == "checksum":
        s["gen"].init()
        return [v.view(torch.int64) for v in s["gen"].generate_checksum(case["rows"])]
    if kind == "resume":
        s["gen"].skip(case["skip"])
        return s["gen"].generate(case["rows"], out=s["out"]).view(torch.int64)
    if kind == "host":
        s["gen"].init()
        return s["gen"].generate_to_host(case["rows"], out=s["out"])
    if kind == "batch":
        here = torch.cuda.current_stream()
        s["batch"].stream.wait_stream(here)
        s["batch"].run()
        here.wait_stream(s["batch"].stream)
        return s["flat"]
    if kind == "noalloc":
        a = s["args"]
        rc = s["lib"].rng_batch_generate_noalloc(case["count"], a[0], a[1], a[2], a[3],
                                                 ctypes.c_void_p(torch.cuda.current_stream().cuda_stream), None)
        if rc:
            raise RuntimeError("rng_batch_generate_noalloc: %d" % rc)
        return s["flat"]
    # serve: the results of the last burst go back first
    server, held = s["server"], s["held"]
    while held:
        server.release(held.pop())
    place = {server.submit(*q): k for k, q in enumerate(s["requests"])}
    outs = [None] * len(place)
    while len(held) < len(place):
        for ticket, addr, _ in server.poll():
            k = place[ticket]
            held.append(ticket)
            key = (addr, k)
            if key not in s["views"]:
                view = torch.as_tensor(_DeviceMemory(addr, s["requests"][k][1] * s["requests"][k][2]), device="cuda")
                view.server = server  # the memory lives as long as the server does
                s["views"][key] = view
            outs[k] = s["views"][key]
    return outs


def work(case):
    """Each output value written once; a generator's states read (when they are
    in memory) and written once.  Per value 6 64-bit operations for the update,
    1 for the stronger output, 2 for a checksum."""
    kind = case["kind"]
    if kind in ("batch", "noalloc", "serve"):
        v = sum(i.streams * i.iterations for i in _instances(case, 0))
        return {"bytes": 8 * v, "flops": 6 * v}
    n, t = case["streams"], case["rows"]
    per = 6 + case["mode"]
    if kind == "checksum":
        return {"bytes": 8 * n + 16 * t, "flops": (per + 2) * n * t}
    state = 16 * n if kind in ("call", "resume") or (kind == "device" and not case["fresh"]) else 8 * n
    return {"bytes": 8 * n * t + state, "flops": per * n * t}


def _shr(x, k):
    return (x >> k) & ((1 << (64 - k)) - 1)


def _step(s):
    s = s ^ (s << 21)
    s = s ^ _shr(s, 35)
    return s ^ (s << 4)


def _first(n, seed, dev):
    """The states that the streams start from: the paper's hash of the id."""
    m, lo = seed & _M64, 0xFFFFFFFF
    m = ((m ^ (m >> 30)) * 0xBF58476D1CE4E5B9) & _M64
    m = ((m ^ (m >> 27)) * 0x94D049BB133111EB) & _M64
    m ^= m >> 31
    a = torch.arange(n, dtype=torch.int64, device=dev) ^ ((m ^ (m >> 32)) & lo)
    a = ((a + 0x7ED55D16) + (a << 12)) & lo
    a = (a ^ 0xC761C23C) ^ (a >> 19)
    a = ((a + 0x165667B1) + (a << 5)) & lo
    a = ((a + 0xD3A2646C) ^ (a << 9)) & lo
    a = ((a + 0xFD7046C5) + (a << 3)) & lo
    a = (a ^ 0xB55A4F09) ^ (a >> 16)
    b = (a ^ 61) ^ (a >> 16)
    b = (b + (b << 3)) & lo
    b = b ^ (b >> 4)
    b = (b * 0x27D4EB2D) & lo
    b = b ^ (b >> 15)
    return (b << 32) | a


def _rows(n, seed, t, mode=0):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    out = torch.empty((t, n), dtype=torch.int64, device=dev)
    s = _first(n, seed, dev)
    for i in range(t):
        out[i] = s * 0x2545F4914F6CDD1D if mode else s
        s = _step(s)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "resume":
        return None  # stepping that far takes too long
    if kind in ("batch", "noalloc", "serve"):
        insts = _instances(case, seed)
        if sum(i.iterations for i in insts) > 20000:
            return None
        outs = [_rows(i.streams, i.seed, i.iterations).reshape(-1) for i in insts]
        if kind == "serve":
            return outs
        offs, total = _offsets(insts)
        flat = torch.zeros(total, dtype=torch.int64, device=outs[0].device)
        for o, v in zip(offs, outs):
            flat[o:o + v.numel()] = v
        return flat
    n, t, mode = case["streams"], case["rows"], case["mode"]
    if t > 70000 or n * t > 1 << 33:
        return None
    if kind == "checksum":
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        xs, ss, s = [], [], _first(n, seed, dev)
        for _ in range(min(t, 2048)):
            e = s * 0x2545F4914F6CDD1D if mode else s
            ss.append(e.sum())
            while e.numel() > 1:
                h = e.numel() // 2
                e = torch.cat([e[:h] ^ e[h:2 * h], e[2 * h:]])
            xs.append(e.reshape(()))
            s = _step(s)
        return [torch.stack(xs), torch.stack(ss)] if t <= 2048 else None
    skipped = kind == "device" and not case["fresh"]
    out = _rows(n, seed, t + skipped, mode)
    return out[1:] if skipped else out
