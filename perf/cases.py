"""The k-mer counting work this library is timed on.

Every case simulates reads on the GPU from a seed (a uniform genome with the
repeats, GC content, read lengths, strands and error rates of the repository's
own workloads in ``datagen``) and counts them through one public entry point:

  device   ``Context.count_device`` on device-resident reads, the result copied
           into the caller's tensors with ``hsk_result_copy``
  host     ``Context.count`` on page-locked host reads
  batch    ``Context.count_batch`` on several host-resident read sets
  ext      ``Context.count_ext``: the counts with every kept k-mer's
           occurrences (read, position)

The caller's result buffers have a capacity that the case alone decides; the
entries past the result stay zero.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

import paper_2407_07718_gb300 as hsk

HIST_LEN = 65536  # the context's default number of histogram bins
CHUNK = 1 << 26   # bases simulated at a time
LONG_MEAN, LONG_SD, LONG_MIN = 10_000, 4_000, 1_000  # log-normal long reads


def _case(name, call, reads, genome, coverage, k, m, lo, hi, **more):
    c = dict(name=name, call=call, reads=reads, genome=genome, coverage=coverage, k=k, m=m, lo=lo, hi=hi,
             read_len=150, sub=0.01, n_rate=0.0, repeats=0, gc=0.0, sets=1)
    if reads == "long":
        c.update(sub=0.005)
    c.update(more)
    return c


def listed():
    return [
        # the smallest job a program sends: 2,000 short reads (a spot check, a
        # plasmid, the tail of a sample); launches and host reads dominate
        _case("device_2k_reads_k31", "device", "short", 1_000_000, 0.3, 31, 17, 2, 1000),
        # a small sample: 20,000 short reads of a 1 Mbp genome
        _case("device_20k_reads_k31", "device", "short", 1_000_000, 3.0, 31, 17, 2, 1000),
        # an ordinary served request: a bacterial genome, short reads, k = 21
        _case("device_request_k21", "device", "short", 2_000_003, 20.0, 21, 11, 2, 1000),
        # an ordinary served request with 10 kb reads and 128-bit keys, ragged size
        _case("device_request_long_k55", "device", "long", 2_345_679, 17.3, 55, 21, 2, 1000),
        # a tenth of the long-read workload: repeats, 30x, [2, 8] filter
        _case("device_long_5mbp_k31", "device", "long", 5_000_000, 30.0, 31, 17, 2, 8, repeats=20),
        # low coverage with every k-mer kept (lo = 1): few copies, many output pairs
        _case("device_keep_all_k31", "device", "short", 20_000_000, 8.0, 31, 17, 1, 1 << 20, read_len=151),
        # the flagship long-read workload: 1.5 G windows of 64-bit keys
        _case("device_long_50mbp_k31", "device", "long", 50_000_000, 30.0, 31, 17, 2, 8, repeats=20),
        # the flagship short-read workload: 2 Gbp, 128-bit keys, N bases, a GC-rich segment
        _case("device_short_100mbp_k55", "device", "pairs", 100_000_000, 20.0, 55, 21, 2, 500, n_rate=1e-4, gc=0.6),
        # reads in host memory, copies inside the call, results back on the host
        _case("host_long_10mbp_k31", "host", "long", 10_000_000, 30.0, 31, 17, 2, 8, repeats=4),
        # many small read sets counted by one call
        _case("batch_10_sets_k31", "batch", "short", 1_500_000, 25.0, 31, 17, 2, 1000, sets=10),
        # counting for seed-and-extend overlap detection: occurrence lists too
        _case("ext_long_5mbp_k31", "ext", "long", 5_000_000, 30.0, 31, 17, 2, 8, repeats=20),
    ]


def draw(rng):
    call = rng.choices(["device", "host", "batch", "ext"], [7, 1, 1, 1])[0]
    reads = rng.choice(["short", "pairs", "long"])
    k = rng.choice([21, 31, 55, rng.randint(17, 32), rng.randint(33, 63)])
    m = {21: 11, 31: 17, 55: 21}.get(k, rng.randint(11, min(k - 5, 23)))
    coverage = round(math.exp(rng.uniform(math.log(4.0), math.log(60.0))), 2)
    top = {"device": 1.2e9, "host": 4e8, "batch": 4e7, "ext": 2e8}[call]
    bases = math.exp(rng.uniform(math.log(3e5), math.log(top)))
    genome = max(30_000, int(bases / coverage)) | 1
    lo = rng.choice([1, 2, 2, 3])
    hi = rng.choice([8, 50, 500, 1000])
    more = dict(read_len=rng.randint(100, 251), n_rate=rng.choice([0.0, 1e-4]),
                repeats=rng.choice([0, 0, 4, 20]) if genome >= 2_000_000 else 0, gc=rng.choice([0.0, 0.6]))
    if call == "batch":
        more["sets"] = rng.randint(3, 10)
    c = _case("", call, reads, genome, coverage, k, m, lo, hi, **more)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# reads, simulated on the GPU
# ---------------------------------------------------------------------------
def _genome(case, size, g):
    bases = torch.randint(0, 4, (size,), generator=g, device="cuda", dtype=torch.uint8)
    if case["gc"]:  # a fifth of the genome at another GC content
        a, n = size // 5, size // 5
        gc = torch.rand(n, generator=g, device="cuda") < case["gc"]
        low = bases[a:a + n] & 1
        bases[a:a + n] = torch.where(gc, 1 + low, 3 * low)  # C/G or A/T
    for _ in range(case["repeats"]):  # families of diverged copies
        n = int(1000 * 20 ** float(torch.rand(1, generator=g, device="cuda")))
        n = min(n, size // 100)
        copies = 100 if size >= 5_000_000 else 20
        fam = torch.randint(0, 4, (n,), generator=g, device="cuda", dtype=torch.uint8)
        div = 0.02 * torch.rand(copies, 1, generator=g, device="cuda")
        hit = torch.rand(copies, n, generator=g, device="cuda") < div
        add = torch.randint(1, 4, (copies, n), generator=g, device="cuda", dtype=torch.uint8)
        fam = (fam[None, :] + hit * add) & 3
        at = torch.randint(0, size - n, (copies,), generator=g, device="cuda")
        for c, p in enumerate(at.tolist()):
            bases[p:p + n] = fam[c]
    return bases


def _reads(case, size, coverage, seed):
    """(ASCII bases uint8, offsets int64) of one read set, on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed & 0x7FFFFFFFFFFFFFFF)
    genome = _genome(case, size, g)
    L = case["read_len"]
    if case["reads"] == "long":
        s2 = math.log(1 + (LONG_SD / LONG_MEAN) ** 2)
        n = max(1, round(size * coverage / LONG_MEAN))
        lens = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
        lens = (lens * math.sqrt(s2) + math.log(LONG_MEAN) - s2 / 2).exp().long().clamp(LONG_MIN, size // 2)
    else:
        n = max(2, round(size * coverage / L))
        n += n & 1
        lens = torch.full((n,), L, device="cuda", dtype=torch.int64)
    room = (size - lens - 2).clamp(min=1)
    start = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * room).long()
    flip = torch.rand(n, generator=g, device="cuda") < 0.5
    if case["reads"] == "pairs":  # mate 2 is the other end of the fragment, on the other strand
        frag = (400 + 50 * torch.randn(n // 2, generator=g, device="cuda")).long().clamp(min=L)
        start[1::2] = torch.minimum(start[0::2] + frag - L, room[1::2])
        flip[1::2] = ~flip[0::2]
    offs = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    torch.cumsum(lens, 0, out=offs[1:])
    total = int(offs[-1])
    out = torch.empty(total, device="cuda", dtype=torch.uint8)
    letters = torch.tensor(list(b"ACGT"), device="cuda", dtype=torch.uint8)
    p_ins = p_del = 0.0005 if case["reads"] == "long" else 0.0
    cuts = [0]
    if total > CHUNK:
        cuts += torch.searchsorted(offs, torch.arange(CHUNK, total, CHUNK, device="cuda")).tolist()
    cuts += [n]
    for r0, r1 in zip(cuts[:-1], cuts[1:]):
        if r1 <= r0:
            continue
        b0, b1 = int(offs[r0]), int(offs[r1])
        read = torch.repeat_interleave(torch.arange(r0, r1, device="cuda"), lens[r0:r1], output_size=b1 - b0)
        at = torch.arange(b0, b1, device="cuda") - offs[read]  # position in the read
        if p_ins:
            r = torch.rand(b1 - b0, generator=g, device="cuda")
            ins = r < p_ins
            step = torch.cumsum((r > 1 - p_del).int() - ins.int(), 0)
            at = (at + step - step[offs[read] - b0]).clamp(min=0)
        back = flip[read]
        pos = start[read] + torch.where(back, lens[read] - 1 - at, at)
        base = genome[pos.clamp(0, size - 1)]
        base = torch.where(back, 3 - base, base)
        r = torch.rand(b1 - b0, generator=g, device="cuda")
        err = r < case["sub"]
        if p_ins:
            err |= ins
        add = torch.randint(1, 4, (b1 - b0,), generator=g, device="cuda", dtype=torch.uint8)
        base = torch.where(err, (base + add) & 3, base)
        text = letters[base.long()]
        if case["n_rate"]:
            text[torch.rand(b1 - b0, generator=g, device="cuda") < case["n_rate"]] = ord("N")
        out[b0:b1] = text
    return out, offs


def _read_sets(case, seed):
    return [_reads(case, size, coverage, seed * 1009 + i) for i, (size, coverage) in enumerate(_set_list(case))]


def _set_list(case):
    """(genome size, coverage) of every read set: a batch's sizes are spread over
    a decade up to case["genome"], its coverages around case["coverage"]."""
    n = case["sets"]
    if case["call"] != "batch":
        return [(case["genome"], case["coverage"])]
    return [(max(20_000, int(case["genome"] * 10 ** (-i / max(n - 1, 1)))), case["coverage"] * (0.6 + 0.8 * (i % 4) / 3))
            for i in range(n)]


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h.numpy()


# ---------------------------------------------------------------------------
# the caller's result buffers
# ---------------------------------------------------------------------------
SCALARS = ("n_windows", "n_distinct", "max_count")


def _capacity(case, size, coverage):
    """Pairs a result buffer holds: the genome's k-mers and the errors seen lo times."""
    L = LONG_MEAN if case["reads"] == "long" else case["read_len"]
    windows = size * coverage * 1.1 * max(L - case["k"] + 1, 1) / L + 4096
    wrong = windows * (1.1 - (1 - 1.3 * case["sub"]) ** case["k"])
    return int(min(windows, size + (wrong if case["lo"] <= 1 else 0.1 * windows))) + 4096


def _buffers(case, cap, empty):
    kw = 1 if case["k"] <= 32 else 2
    out = {"kmers": empty((cap, kw), "int64"), "counts": empty((cap,), "int32"), "hist": empty((HIST_LEN,), "int64")}
    if case["call"] == "ext":
        occ = cap * (min(case["hi"], 64) if case["lo"] > 1 else 4)
        out.update(occ_offsets=empty((cap + 1,), "int64"), occ_read=empty((occ,), "int32"), occ_pos=empty((occ,), "int32"))
    return out


def _all_buffers(case):
    """One set of zeroed buffers for each read set; on the device for device calls."""
    if case["call"] == "device":
        def empty(shape, t):
            return torch.zeros(shape, dtype=getattr(torch, t), device="cuda")
    else:
        def empty(shape, t):
            a = np.empty(shape, t)
            a.fill(0)
            return a
    return [_buffers(case, _capacity(case, s, c), empty) for s, c in _set_list(case)]


def prepare(case, seed):
    sets = _read_sets(case, seed)
    state = {"case": case, "ctx": hsk.Context(device=torch.cuda.current_device()), "out": _all_buffers(case)}
    if case["call"] == "device":
        state["reads"], state["offsets"] = sets[0]
    else:  # host arrays a program has read its files into, page-locked as bench.py's are
        state["host"] = [(_pinned(r), _pinned(o).view(np.uint64)) for r, o in sets]
    torch.cuda.synchronize()
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _device_result(ctx, r, out):
    """The counts of a count_device call in the caller's device tensors."""
    n = int(r.n_pairs)
    if n > out["counts"].numel():
        raise ValueError("result buffers too small")
    stream = torch.cuda.current_stream().cuda_stream
    rc = ctx.lib.hsk_result_copy(ctx.h, ctypes.byref(r), out["kmers"].data_ptr(), out["counts"].data_ptr(),
                                 out["hist"].data_ptr(), 1, stream)
    if rc != hsk.HSK_OK:
        raise hsk.HskError(rc, ctx.lib.hsk_last_error(ctx.h).decode())
    return {**out, **{f: int(getattr(r, f)) for f in SCALARS}}


def _fill(dst, src):
    dst[: len(src)] = src.view(dst.dtype).reshape((len(src),) + dst.shape[1:])


def _host_result(r, out):
    for f in ("kmers", "counts", "hist"):
        _fill(out[f], getattr(r, f))
    return {**out, **{f: int(getattr(r, f)) for f in SCALARS}}


def run(state):
    case, ctx, out = state["case"], state["ctx"], state["out"]
    args = case["k"], case["m"], case["lo"], case["hi"]
    if case["call"] == "device":
        return _device_result(ctx, ctx.count_device(state["reads"], state["offsets"], *args), out[0])
    if case["call"] == "host":
        return _host_result(ctx.count(*state["host"][0], *args, copy="view"), out[0])
    if case["call"] == "batch":
        got = ctx.count_batch([(r, o, *args) for r, o in state["host"]], copy="view")
        return [_host_result(r, o) for r, o in zip(got, out)]
    r, off, read, pos = ctx.count_ext(*state["host"][0], *args)
    for f, a in (("occ_offsets", off), ("occ_read", read), ("occ_pos", pos)):
        _fill(out[0][f], a)
    return _host_result(r, out[0])


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _set_bytes(case, size, coverage):
    L = LONG_MEAN if case["reads"] == "long" else case["read_len"]
    n_reads, k = size * coverage / L, case["k"]
    good = (1 - case["sub"]) ** k
    windows = n_reads * max(L - k + 1, 0)
    lam = windows / size * good  # error-free copies of a genome k-mer, Poisson
    lo, hi = case["lo"], min(case["hi"], int(lam + 20 * math.sqrt(lam) + 50))
    p = sum(math.exp(-lam + c * math.log(lam) - math.lgamma(c + 1)) for c in range(lo, hi + 1)) if lam > 0 else 0.0
    kept = size * p + (windows * (1 - good) if lo <= 1 else 0)
    pair = (8 if k <= 32 else 16) + 4
    occ = 0.0
    if case["call"] == "ext":  # (read, position) of every occurrence, one offset per kept k-mer
        occ = kept * (8 + 8 * max(lo, min(lam, hi)))
    return size * coverage + 8 * n_reads + kept * pair + occ + 8 * HIST_LEN


def work(case):
    return {"bytes": int(sum(_set_bytes(case, s, c) for s, c in _set_list(case))), "flops": 0}


# ---------------------------------------------------------------------------
# the same counts from plain tensor operations
# ---------------------------------------------------------------------------
_SIGN = -(1 << 63)


def _code(base, n, rc):
    """2-bit code of the n <= 32 bases (or their reverse complement) from every position."""
    def join(a, na, b, nb):  # bases [i, i + na) then [i + na, i + na + nb)
        a, b = a[: a.numel() - nb], b[na:]
        return (b << (2 * na)) | a if rc else (a << (2 * nb)) | b
    part, size, out, done = (3 - base if rc else base).long(), 1, None, 0
    while True:
        if n & size:
            out, done = (part, size) if out is None else (join(out, done, part, size), done + size)
        if size * 2 > n:
            return out
        part, size = join(part, size, part, size), size * 2


def _exact_set(case, reads, offs):
    k, dev = case["k"], reads.device
    codes = torch.full((256,), 4, dtype=torch.uint8, device=dev)
    codes[torch.tensor(list(b"ACGT"), device=dev)] = torch.arange(4, dtype=torch.uint8, device=dev)
    base = codes[reads.long()]
    n = base.numel() - k + 1
    bad = torch.zeros(base.numel() + 1, dtype=torch.int32, device=dev)
    torch.cumsum(base == 4, 0, out=bad[1:])
    ok = bad[k:] == bad[:-k]
    starts = torch.zeros(base.numel() + 1, dtype=torch.int32, device=dev)
    starts[offs[:-1]] = 1
    inner = torch.cumsum(starts, 0)
    ok &= inner[k - 1: k - 1 + n] == inner[:n]  # no read starts inside the window
    base = base & 3
    where = torch.nonzero(ok).squeeze(1)
    del bad, starts, inner, ok
    if k <= 32:
        f, r = _code(base, k, False)[where] ^ _SIGN, _code(base, k, True)[where] ^ _SIGN
        keys, counts = torch.unique(torch.minimum(f, r), return_counts=True)
        kmers = (keys ^ _SIGN)[:, None]
    else:
        h = k - 32  # {lo, hi}: the last 32 bases and the h before them
        fh, fl = _code(base, h, False)[where] ^ _SIGN, _code(base, 32, False)[where + h] ^ _SIGN
        rh, rl = _code(base, h, True)[where + 32] ^ _SIGN, _code(base, 32, True)[where] ^ _SIGN
        fwd = (fh < rh) | ((fh == rh) & (fl <= rl))
        hi, lo = torch.where(fwd, fh, rh), torch.where(fwd, fl, rl)
        del fh, fl, rh, rl, fwd
        lo, order = torch.sort(lo, stable=True)
        hi, order2 = torch.sort(hi[order], stable=True)
        lo = lo[order2]
        del order, order2
        new = torch.ones(hi.numel(), dtype=torch.bool, device=dev)
        new[1:] = (hi[1:] != hi[:-1]) | (lo[1:] != lo[:-1])
        at = torch.nonzero(new).squeeze(1)
        counts = torch.diff(at, append=torch.tensor([hi.numel()], device=dev))
        kmers = torch.stack([lo[at] ^ _SIGN, hi[at] ^ _SIGN], 1)
    hist = torch.bincount(counts.clamp(max=HIST_LEN - 1), minlength=HIST_LEN)
    keep = (counts >= case["lo"]) & (counts <= case["hi"])
    return {"kmers": kmers[keep], "counts": counts[keep].int(), "hist": hist, "n_windows": int(where.numel()),
            "n_distinct": int(counts.numel()), "max_count": int(counts.max()) if counts.numel() else 0}


def exact(case, seed):
    if case["genome"] * case["coverage"] * case["sets"] > 4.5e8:
        return None
    results = []
    for reads, buf in zip(_read_sets(case, seed), _all_buffers(case)):
        r = _exact_set(case, *reads)
        for f in ("kmers", "counts", "hist"):
            if case["call"] == "device":
                buf[f][: r[f].shape[0]] = r[f]
            else:
                _fill(buf[f], r[f].cpu().numpy())
        for f in ("occ_offsets", "occ_read", "occ_pos"):
            if f in buf:
                buf[f] = None  # occurrence lists: whole numbers, not recomputed here
        results.append({**buf, **{f: r[f] for f in SCALARS}})
    return results if case["call"] == "batch" else results[0]
