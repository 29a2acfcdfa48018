"""Performance cases of the matched-filter search, through its public entry points.

A pass of a case is what a program that keeps a context and a template bank
does with one more piece of strain: load the segment, correlate it with the
bank, bring sigma and the tails to the host in (template, lag) order, release
the handles.  Strain and results are host data, as they are for such a
program, except in the kind that works on the caller's device buffers.

Kinds ("kind" of a case):
  search  bege_load_segment, bege_correlate / bege_correlate_ex, fetch, release;
          "define" defines the bank in the pass as well (a follow-up search
          makes its own bank), "ex" runs the overlap-save mask with the
          per-lag maximum, "precision" selects the context's arithmetic
  device  bege_search_noalloc on device buffers of the caller
  block   bege_correlate_multi: one bank against several segments
  batch   bege_batch_run of a prepared batch of unequal segments, results fetched
  serve   requests submitted to a running server and waited for

Strain is unit-variance Gaussian noise limited to 350-2000 Hz at 4096 Hz, with
an injected chirp where a case says so; banks are chirps inside that band, or
plain Gaussian samples.
"""
import math

import numpy as np
import torch

from paper_1708_01609_gb300 import binding

FS = 4096.0
BAND = (350.0, 2000.0)
TAPER = 0.05


def listed():
    return [
        # an alert-sized question: 4 s of strain, the 64-chirp parity bank, one signal;
        # launches, allocations and latency are all of it
        case("alert", "search", 14, 64, 4096, kappa=5.0, inject=1),
        # 1 s of strain against 1000-sample templates given as samples (odd count, one
        # column per transform)
        case("short", "search", 12, 1003, 1000, kappa=5.0, samples=1),
        # 8 s of strain and a half-second bank in a caller's own device memory
        case("device", "device", 15, 5001, 2050),
        # follow-up of a candidate: a fresh bank of 2048 chirps is defined, searched and dropped
        case("followup", "search", 16, 2048, 4096, define=1, inject=1),
        # the benchmark's search: 16 s of strain against the bank of 2^20 one-second chirps
        case("full_bank", "search", 16, 1 << 20, 4096),
        # 32 s of strain, the longest segment, an odd share of a bank
        case("long", "search", 17, 20011, 4096),
        # templates of about 3 s, longer than a column
        case("long_templates", "search", 16, 3001, 12001, samples=1),
        # overlap-save lags with the per-lag maximum over the bank (the first pass's output)
        case("projection", "search", 16, 16384, 4096, ex=1, inject=1),
        # the block form: eight 16 s segments share each template's transform
        case("block", "block", 16, 6000, 4096, segments=8),
        # the batching form: twelve segments of 4 to 32 s, each with a range of its own
        case("batch", "batch", 17, 30000, 4096, segments=12),
        # the tensor-core precision form
        case("bf16x3", "search", 16, 16384, 4096, precision=1),
        # the serving form: six requests of 8, 16 and 32 s from two channels
        case("serve", "serve", 17, 12000, 4096, segments=6),
    ]


def case(name, kind, lg, count, length, kappa=5.5, inject=0, samples=0, define=0, ex=0,
         precision=0, segments=1):
    c = {"name": name, "kind": kind, "lg": lg, "count": count, "length": length, "kappa": kappa,
         "inject": inject, "samples": samples, "define": define, "ex": ex,
         "precision": precision, "segments": segments}
    if not name:
        del c["name"]
    return c


def draw(rng):
    kind = rng.choice(["search"] * 5 + ["device", "block", "batch", "serve"])
    wide = kind in ("search", "device")
    lg = rng.randint(10, 17) if kind == "search" else rng.randint(10, 16) if kind == "device" \
        else rng.randint(14, 17)
    n = 1 << lg
    # correlations of all segments of a case times their length: at most 2^33 samples
    segments = 1 if wide else rng.randint(2, 8) if kind == "block" else rng.randint(3, 12)
    top = min(1 << 18, (1 << 33) // n // (1 if wide else segments))
    count = int(round(math.exp(rng.uniform(math.log(33), math.log(top)))))
    if kind == "serve":
        count = max(count, 1000)
    form = rng.random()
    if wide and form < 0.25:  # templates of any length the segment takes
        length = int(round(math.exp(rng.uniform(math.log(64), math.log(min(n, 1 << 16))))))
        count = min(count, max(33, (1 << 26) // length))
        return case("", kind, lg, count, length, samples=1)
    length = min(n, rng.choice([4096, 4096, 2048, 3000]))
    if kind != "search":
        return case("", kind, lg, count, length, segments=segments)
    if lg >= 14 and form < 0.4:
        return case("", kind, lg, count, length, precision=rng.choice([1, 1, 2]))
    return case("", kind, lg, count, length, kappa=rng.choice([5.0, 5.5, 5.5, 6.0]),
                ex=rng.choice([0, 0, 1]), define=int(count <= 8192 and rng.random() < 0.3))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def noise(n, seed):
    """Band-limited Gaussian noise of unit variance, FP64 host array."""
    rng = np.random.default_rng(seed)
    spec = np.zeros(n // 2 + 1, dtype=np.complex128)
    f = np.arange(n // 2 + 1) * FS / n
    inside = np.nonzero((f >= BAND[0]) & (f <= BAND[1]))[0]
    s = n / math.sqrt(2.0 * len(inside))
    spec[inside] = s * (rng.standard_normal(len(inside)) +
                        1j * rng.standard_normal(len(inside))) * math.sqrt(0.5)
    return np.fft.irfft(spec, n=n)


def chirps(count, tau, seed):
    """`count` chirps (f0, fdot) whose frequency stays in the band over tau seconds."""
    rng = np.random.default_rng(seed)
    fdot = np.sort(rng.uniform(-200.0, 200.0, count))
    low = BAND[0] + np.maximum(0.0, -fdot * tau)
    high = BAND[1] - np.maximum(0.0, fdot * tau)
    return np.stack([low + (high - low) * rng.random(count), fdot], axis=1)


def chirp_rows(params, length, device="cpu"):
    """The chirp templates in FP64: tapered, unit norm."""
    p = torch.as_tensor(params, dtype=torch.float64, device=device)
    t = torch.arange(length, dtype=torch.float64, device=device) / FS
    cycles = p[:, :1] * t + 0.5 * p[:, 1:] * t * t
    m = torch.arange(length, dtype=torch.float64, device=device)
    m = torch.minimum(m, length - 1 - m)
    width = math.floor(TAPER * (length - 1) / 2.0)
    edge = 0.5 * (1.0 - torch.cos(2.0 * math.pi * m / (TAPER * (length - 1))))
    w = torch.sin(2.0 * math.pi * (cycles - torch.floor(cycles))) * \
        torch.where(m <= width, edge, torch.ones_like(edge))
    return w / torch.sqrt((w * w).sum(dim=1, keepdim=True))


def lengths(c):
    """Segment length of each segment of a case (block: equal; batch, serve: 4 to 32 s)."""
    lg, k = c["lg"], c["segments"]
    if c["kind"] in ("batch", "serve"):
        low = 14 if c["kind"] == "batch" else 15
        return [1 << max(low, lg - (i % 4 if c["kind"] == "batch" else i % 3)) for i in range(k)]
    return [1 << lg] * k


def ranges(c):
    """Bank rows [k0, k1) of each segment: a batch cuts unequal ranges of the bank."""
    k, count = c["segments"], c["count"]
    if c["kind"] != "batch":
        return [(0, count)] * k
    cut = [count * i * (i + k) // (2 * k * k) for i in range(k + 1)]
    return [(a, max(a + 1, b)) for a, b in zip(cut, cut[1:])]


def inputs(c, seed):
    """Strain of each segment (FP32), chirp parameters or sample rows (FP32)."""
    tau = c["length"] / FS
    params = rows = None
    if c["samples"] or c["kind"] == "device":
        g = torch.Generator().manual_seed(seed + 17)
        rows = torch.randn(c["count"], c["length"], generator=g)
    else:
        params = chirps(c["count"], tau, seed + 17)
    strain = []
    for i, n in enumerate(lengths(c)):
        y = noise(n, (seed, i))
        if c["inject"]:
            rng = np.random.default_rng((seed, i, 5))
            k = int(rng.integers(c["count"]))
            at = int(rng.integers(n - c["length"] + 1))
            y[at:at + c["length"]] += rng.uniform(8.0, 12.0) * math.sqrt(
                n / (2.0 * np.count_nonzero((np.arange(n // 2 + 1) * FS / n >= BAND[0]) & (
                    np.arange(n // 2 + 1) * FS / n <= BAND[1])))) * \
                chirp_rows(params[k:k + 1], c["length"])[0].numpy()
        strain.append(y.astype(np.float32))
    return strain, params, rows


class State:
    """What the program keeps: its context, bank, strain and the form's handle."""


def prepare(c, seed):
    s = State()
    s.c, s.tau = c, c["length"] / FS
    s.strain, s.params, rows = inputs(c, seed)
    if c["kind"] == "device":
        ld = (c["length"] + 7) // 8 * 8
        s.ld = ld
        s.bank = torch.zeros(c["count"], ld, device="cuda")
        s.bank[:, :c["length"]] = rows.cuda()
        s.y = torch.from_numpy(s.strain[0]).cuda()
        s.sigma = torch.empty(c["count"], device="cuda")
        s.recs = torch.empty(1 << 20, 3, dtype=torch.int32, device="cuda")
        s.total = torch.zeros(1, dtype=torch.int64, device="cuda")
        return s
    s.ctx = binding.Context(0, fs=FS, precision=c["precision"])
    if not c["define"]:
        s.bank = (s.ctx.bege_define_bank_samples(rows.numpy()) if c["samples"] else
                  s.ctx.bege_define_bank(s.params, tau=s.tau, taper_frac=TAPER))
    if c["kind"] == "batch":
        s.batch = s.ctx.bege_batch_create(
            [(y, s.bank, k0, k1, c["kappa"]) for y, (k0, k1) in zip(s.strain, ranges(c))],
            tail_capacity=1 << 18)
    if c["kind"] == "serve":
        s.server = s.ctx.bege_serve_create(s.bank, c["kappa"], slice_templates=4096)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def buffer(c, n, rows):
    """Room for the tails of one segment: four times what noise gives, and what a signal
    lights up in the bank."""
    noise_tails = n * rows * math.erfc(c["kappa"] / math.sqrt(2.0))
    return 1 << int(512 + 4 * noise_tails + c["inject"] * (2048 + 2 * rows)).bit_length()


def found(c, n, rows, recs, sigma, total):
    """The tails in the program's own table, zero beyond them, with their number and sigma."""
    table = np.zeros((3, buffer(c, n, rows)), dtype=np.int32)
    m = min(len(recs), table.shape[1])
    table[0, :m], table[1, :m] = recs["tmpl"][:m], recs["lag"][:m]
    value = table[2].view(np.float32)
    value[:m] = recs["value"][:m]
    return {"tmpl": table[0], "lag": table[1], "value": value, "sigma": sigma, "total": total}


def run(s):
    c = s.c
    if c["kind"] == "device":
        binding.bege_search_noalloc(s.y.data_ptr(), len(s.y), s.bank.data_ptr(), s.ld, 0,
                                    c["count"], c["kappa"], s.sigma.data_ptr(),
                                    s.recs.data_ptr(), len(s.recs), s.total.data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
        total = int(s.total.item())
        recs = s.recs[:total].cpu().numpy().reshape(-1).view(binding.TAIL_DTYPE)
        return found(c, len(s.y), c["count"], binding.bege_sort_tails(recs), s.sigma, total)
    ctx = s.ctx
    if c["kind"] == "batch":
        ctx.bege_batch_run(s.batch)
        out = []
        for i, (k0, k1) in enumerate(ranges(c)):
            recs, total = ctx.bege_batch_fetch_tails(s.batch, i)
            sigma = ctx.bege_batch_get_sigma(s.batch, i, k1 - k0)
            out.append(found(c, len(s.strain[i]), k1 - k0, binding.bege_sort_tails(recs), sigma,
                             total))
        return out
    if c["kind"] == "serve":
        ids = [ctx.bege_serve_submit(s.server, y, i % 2) for i, y in enumerate(s.strain)]
        out = []
        for y, r in zip(s.strain, ids):
            ctx.bege_serve_wait(s.server, r)
            recs, total = ctx.bege_serve_fetch_tails(s.server, r)
            sigma = ctx.bege_serve_get_sigma(s.server, r, c["count"])
            out.append(found(c, len(y), c["count"], binding.bege_sort_tails(recs), sigma, total))
            ctx.bege_serve_forget(s.server, r)
        return out
    bank = s.bank if not c["define"] else ctx.bege_define_bank(s.params, tau=s.tau,
                                                               taper_frac=TAPER)
    segs = [ctx.bege_load_segment(y) for y in s.strain]
    if c["kind"] == "block":
        jobs = ctx.bege_correlate_multi(segs, bank, 0, c["count"], c["kappa"])
    elif c["ex"]:
        jobs = [ctx.bege_correlate_ex(segs[0], bank, 0, c["count"], c["kappa"], linear=True,
                                      project=True)]
    else:
        jobs = [ctx.bege_correlate(segs[0], bank, 0, c["count"], c["kappa"])]
    out = []
    for j in jobs:
        recs, total = ctx.bege_fetch_tails(j, sort=True)
        sigma = ctx.bege_get_sigma(j, c["count"])
        out.append(found(c, len(s.strain[0]), c["count"], recs, sigma, total))
        if c["ex"]:
            snr, best = ctx.bege_fetch_max(j, len(s.strain[0]))
            out[-1].update(snr=snr, best=best)
        ctx.bege_release(j)
    for g in segs:
        ctx.bege_release(g)
    if c["define"]:
        ctx.bege_release(bank)
    return out if c["kind"] == "block" else out[0]


# ---------------------------------------------------------------------------
# What a pass cannot do without, and how exact it is
# ---------------------------------------------------------------------------
def work(c):
    """Bytes: the strain and the bank read once (a range of it for each segment of a batch;
    once for a block), sigma written.  Flops: 5 N log2 N per correlation, the usual count for
    the two real transforms of a matched filter.  Defined banks are written as well."""
    ns, rs = lengths(c), ranges(c)
    rows = sum(b - a for a, b in rs) if c["kind"] == "batch" else c["count"]
    if c["kind"] == "serve":
        rows *= len(ns)
    pairs = sum((b - a) for a, b in rs)
    bytes_ = 4 * sum(ns) + 4 * c["length"] * rows * (2 if c["define"] else 1) + 4 * pairs
    return {"bytes": bytes_, "flops": sum(5.0 * n * math.log2(n) * (b - a)
                                          for n, (a, b) in zip(ns, rs))}


def tolerance(c):
    # against FP64, the FP32 transforms show 1e-7 to 5e-7 (sigma, values) and the split 16-bit
    # operands 5e-7 to 2e-6, with single values five times that; "differ" allows ties of the
    # per-lag maximum
    if c["precision"]:
        return {"rel": 1e-5, "max": 1e-4, "differ": 2e-3}
    return {"rel": 2e-6, "max": 1e-5, "differ": 2e-3}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------
def exact(c, seed):
    pairs = sum((b - a) * n for n, (a, b) in zip(lengths(c), ranges(c)))
    if pairs > 1 << 33:
        return None
    strain, params, rows = inputs(c, seed)
    out = [search64(c, y, params, rows, k0, k1) for y, (k0, k1) in zip(strain, ranges(c))]
    return out if c["kind"] in ("block", "batch", "serve") else out[0]


def search64(c, y, params, rows, k0, k1):
    n, length, dev = len(y), c["length"], "cuda"
    spec = torch.fft.rfft(torch.from_numpy(y).to(dev).double())
    step = max(1, (1 << 24) // n)
    values, sigma = [], []
    snr = torch.zeros(n, dtype=torch.float64, device=dev)
    for a in range(k0, k1, step):
        b = min(k1, a + step)
        w = rows[a:b].to(dev).double() if rows is not None else chirp_rows(params[a:b], length,
                                                                           dev)
        rho = torch.fft.irfft(torch.conj(torch.fft.rfft(w, n=n)) * spec, n=n)
        sig = torch.sqrt((rho * rho).mean(dim=1))
        thr = c["kappa"] * sig[:, None]
        hit = rho.abs() > thr
        if c["ex"]:  # lags whose template window stays inside the segment
            hit &= torch.arange(n, device=dev) <= n - length
            v = torch.where(hit & (rho > thr), rho / sig[:, None], torch.zeros_like(rho))
            snr = torch.maximum(snr, v.max(dim=0).values)
        at = torch.nonzero(hit)
        values.append(rho[at[:, 0], at[:, 1]])
        sigma.append(sig)
    value = torch.zeros(buffer(c, n, k1 - k0), dtype=torch.float64, device=dev)
    found_ = torch.cat(values)[:len(value)]
    value[:len(found_)] = found_
    out = {"tmpl": None, "lag": None, "value": value, "sigma": torch.cat(sigma), "total": None}
    if c["ex"]:
        out.update(snr=snr, best=None)
    return out
