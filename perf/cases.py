"""The work that users of this library have it do, as measurable cases.

Every case is a whole call sequence through the Python binding: a chunk (or several) of an 8-bit
filterbank goes through a plan's dedispersion and single-pulse search and its candidates come back
to the host; or device series go through the allocation-free search; or a batch of beams runs one
step. The sizes are those of this repository's workloads (``synth/configs.py``), its smoke run,
its parity tests and its benchmark.

Plans are streams: a state is primed with as many chunks as the plan's overlap needs, and each
pass delivers the same chunk again, so that every pass computes the same full window. Candidate
times are returned relative to the first sample of the pass.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2101_00941_gb300 as dd

K_DM = 4.148808e3  # s MHz^2 pc^-1 cm^3

MID = "0:0.1:1500:1,150:0.2:750:2,300:0.25:800:4,500:0.5:1000:8"
OOC = MID + ",1000:1.0:2000:16"
MID_500 = "0:0.1:1500:1,150:0.2:750:2,300:0.25:800:4"
W256 = "1,2,4,8,16,32,64,128,256"
W512 = W256 + ",512"


def _case(name, **kw):
    """A beam case: `chunks` chunks of `n` samples a pass through one plan of `streams` streams.
    where: device, pinned or pageable chunks; search: window, clipped or fused."""
    c = dict(name=name, kind="beam", nchans=4096, fch1=1550.0, bw=300.0, tsamp=64e-6, ranges=MID,
             n=1 << 17, chunks=1, streams=1, widths=W256, threshold=6.0, block=32,
             where="device", search="window", pulses=5)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call in use: a few hundred channels, a short chunk, two short DM ranges (the
        # smoke run's beam), where launches and host time count
        _case("small_256ch_8192", nchans=256, bw=75.0, ranges="0:0.0625:70:1,4.375:0.125:40:2",
              n=8192, pulses=2),
        # a small survey's beam with coarse channels, read from pinned host memory (the 64-channel
        # 65536-sample workload)
        _case("tiny_64ch_65536", nchans=64, fch1=1500.0, bw=100.0, ranges="0:1.0:401:1", n=65536,
              widths="1,2,4,8,16,32", where="pinned", pulses=3),
        # the headline beam: one chunk of the 4096-channel, 4050-trial stream, resident on the GPU
        _case("mid_4096ch_131072"),
        # the same stream as it arrives: chunks of 2^16 samples in pinned host memory over four
        # CUDA streams, collected at the end (the serving chunk size)
        _case("stream_4096ch_4x65536", n=65536, chunks=4, streams=4, where="pinned"),
        # a chunk of the out-of-core beam: 8192 channels over 500 MHz, DM 0-3000, x1 .. x16
        _case("ooc_8192ch_262144", nchans=8192, fch1=1500.0, bw=500.0, tsamp=50e-6, ranges=OOC,
              n=1 << 18, widths=W512),
        # a ragged beam: channel count, trial counts and window length that fit no tile, odd
        # widths, decimation up to x32, pageable input
        _case("ragged_1001ch_49984", nchans=1001, bw=1001 * 300.0 / 4096,
              ranges="0:0.1:333:1,33.3:0.2:130:2,60:0.5:65:4,95:1.0:41:32", n=49984,
              widths="1,3,6,12,24,100,256", where="pageable"),
        # a wide, coarse-channel band (256 channels of 1.5625 MHz), DM 0-800
        _case("coarse_256ch_131072", nchans=256, fch1=1500.0, bw=400.0,
              ranges="0:0.5:800:1,400:1.0:400:2", n=1 << 17),
        # one narrow DM search around a known source: few trials, long chunk
        _case("followup_1024ch_96x262144", nchans=1024, fch1=1450.0, bw=200.0,
              ranges="180:0.1:96:1", n=1 << 18, widths="1,2,4,8,16,32,64", block=8),
        # the robust (clipped) noise statistic on a 1024-channel beam
        _case("clipped_1024ch_65536", nchans=1024, fch1=1450.0, bw=200.0, ranges=MID_500, n=65536,
              search="clipped"),
        # the search fused into dedispersion, series not kept
        _case("fused_1024ch_65536", nchans=1024, fch1=1450.0, bw=200.0, ranges=MID_500, n=65536,
              search="fused"),
        # three beams of uneven length and channel count in one captured step
        dict(name="batch_3beams_2e17", kind="batch", chans="1024,4096,1024",
             lens="131072,75008,240128", ranges=MID_500, n=1 << 17, widths=W256, threshold=6.0,
             persistent=False, pulses=5),
        # the search alone, on series a host program already holds
        dict(name="search_750x131072", kind="static", trials=750, n=131072, d=1, widths=W256,
             threshold=6.0, block=32),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["beam"] * 8 + ["static"])
    if kind == "static":
        n, trials = int(_log(rng, 4096, 200000)), int(_log(rng, 16, 2000))
        return dict(kind="static", trials=trials, n=n, d=rng.choice([1, 2, 4]),
                    widths=rng.choice([W256, W512, "1,2,4,8,16,32", "4,12,20,100"]),
                    threshold=6.0, block=rng.choice([8, 32]))
    nchans = int(_log(rng, 64, 4096))
    if rng.random() < 0.5:
        nchans = max(64, nchans // 16 * 16)
    coarse = rng.random() < 0.25  # channels of about 1 MHz, else of the 4096-channel beam's width
    if coarse:
        nchans = min(nchans, 400)
    bw = nchans * (rng.uniform(0.6, 1.6) if coarse else rng.uniform(0.05, 0.2) * (1024 / max(
        nchans, 1024)))
    fch1 = rng.choice([1450.0, 1500.0, 1550.0])
    tsamp = rng.choice([50e-6, 64e-6])
    span = K_DM * ((fch1 - bw) ** -2 - fch1 ** -2) / tsamp  # band delay in samples per unit of DM
    nr = rng.choice([1, 1, 2, 3])
    rows, dm, d = [], rng.choice([0.0, 0.0, 100.0]), 1
    for _ in range(nr):
        ntr = int(_log(rng, 24, 1200))
        step = round(rng.uniform(0.6, 2.5) * d / span, 4)  # band delay per trial, decimated samples
        # keep the overlap of a range below about 30000 samples
        ntr = max(8, min(ntr, int((30000 / span - dm) / step)))
        rows.append("%r:%r:%d:%d" % (round(dm, 4), step, ntr, d))
        dm += ntr * step
        d *= rng.choice([2, 2, 4])
    dmax = 16
    n = int(_log(rng, 8192, 200000)) // dmax * dmax
    adds = nchans * sum(int(r.split(":")[2]) * n // int(r.split(":")[3]) for r in rows)
    if adds > 4e11:
        n = max(8192, int(n * 4e11 / adds) // dmax * dmax)
    return {k: v for k, v in _case(
        "", nchans=nchans, fch1=fch1, bw=bw, tsamp=tsamp, ranges=",".join(rows), n=n,
        streams=1, widths=rng.choice([W256, "1,2,4,8,16,32", "1,3,6,12,24,100"]),
        block=rng.choice([8, 32]), where=rng.choice(["device", "device", "pinned"]),
        search=rng.choice(["window", "window", "clipped", "fused"]), pulses=3).items()
        if k != "name"}


# ---------------------------------------------------------------------------- inputs


def _ranges(text):
    rows = [r.split(":") for r in text.split(",")]
    return [(float(a), float(b), int(c), int(d)) for a, b, c, d in rows]


def _ints(text):
    return [int(w) for w in text.split(",")]


def _freqs(nchans, fch1, bw):
    return fch1 - np.arange(nchans, dtype=np.float64) * (bw / nchans)


def _noise(n, nchans, gen):
    """uint8 [n][nchans] on the GPU: Gaussian noise of mean 128 and deviation 16, clipped."""
    x = torch.empty((n, nchans), dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 26) // nchans)
    for a in range(0, n, step):
        b = min(n, a + step)
        g = torch.randn((b - a, nchans), device="cuda", generator=gen)
        x[a:b] = g.mul_(16.0).add_(128.0).round_().clamp_(0.0, 255.0).to(torch.uint8)
    return x


def _inject(x, freqs, tsamp, dm_max, count, rng):
    """Add dispersed boxcar pulses (DM up to dm_max, width up to 64 samples, SNR 8-30) in place."""
    n, nchans = x.shape
    chans = torch.arange(nchans, device="cuda")
    for _ in range(count):
        dm = rng.uniform(0.0, dm_max)
        width = int(round(math.exp(rng.uniform(0.0, math.log(64.0)))))
        amp = rng.uniform(8.0, 30.0) * 16.0 / math.sqrt(width * nchans)
        delay = K_DM * dm * (freqs ** -2.0 - freqs.max() ** -2.0) / tsamp
        first = torch.from_numpy(np.floor(delay + 0.5).astype(np.int64)).cuda()
        first = first + int(rng.integers(0, n))
        dither = torch.from_numpy(rng.random(nchans)).cuda()
        for k in range(width):
            t = (first + k) % n  # chunks repeat, so a pulse may wrap
            add = torch.floor(amp * (k + 1) + dither) - torch.floor(amp * k + dither)
            v = x[t, chans].double() + add
            x[t, chans] = v.clamp(0.0, 255.0).to(torch.uint8)


def _beam_input(n, freqs, tsamp, ranges, pulses, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = _noise(n, freqs.size, gen)
    dm_max = max(a + b * c for a, b, c, _ in ranges)
    _inject(x, freqs, tsamp, dm_max, pulses, np.random.default_rng(seed))
    return x


def _series_input(case, seed):
    """int32 [trials][n]: what dedispersed noise of 512 channels looks like, with pulses."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    trials, n, d = case["trials"], case["n"], case["d"]
    sd = 16.0 * math.sqrt(512.0 * d)
    y = torch.randn((trials, n), device="cuda", generator=gen).mul_(sd).add_(128.0 * 512 * d)
    rng = np.random.default_rng(seed)
    for _ in range(10):
        w, t, j = int(rng.integers(1, 65)), int(rng.integers(0, trials)), int(rng.integers(0, n))
        y[t, j:j + w] += rng.uniform(8.0, 30.0) * sd / math.sqrt(w)
    return y.round_().clamp_(min=0.0).to(torch.int32)


# ---------------------------------------------------------------------------- prepare, run


class _Owned:
    """A plan's device buffer as a tensor source that keeps the plan alive."""

    def __init__(self, plan, ptr, shape, typestr):
        self.plan = plan
        self.__cuda_array_interface__ = dict(shape=shape, typestr=typestr, data=(ptr, False),
                                             version=3, strides=None)


def _view(plan, ptr, shape, typestr):
    return torch.as_tensor(_Owned(plan, ptr, shape, typestr), device="cuda")


def prepare(case, seed):
    if case["kind"] == "static":
        cap = 1 << 18
        return dict(case=case, y=_series_input(case, seed), cap=cap,
                    widths=_ints(case["widths"]),
                    cands=torch.empty(cap * dd.CAND_DTYPE.itemsize, dtype=torch.uint8,
                                      device="cuda"),
                    count=torch.zeros(1, dtype=torch.int64, device="cuda"))
    ranges, widths = _ranges(case["ranges"]), _ints(case["widths"])
    if case["kind"] == "batch":
        beams = []
        for k, (c, n) in enumerate(zip(_ints(case["chans"]), _ints(case["lens"]))):
            f = _freqs(c, 1550.0, 300.0) if c == 4096 else _freqs(c, 1450.0, 200.0)
            x = _beam_input(n, f, 64e-6, ranges, case["pulses"], seed * 16 + k)
            beams.append((f, 64e-6, x))
        torch.cuda.synchronize()
        b = dd.Batch(beams, ranges, case["n"], widths, case["threshold"], n_streams=2,
                     max_width=max(widths), graph=True, persistent=case["persistent"])
        return dict(case=case, batch=b, beams=beams)
    f = _freqs(case["nchans"], case["fch1"], case["bw"])
    n, chunks = case["n"], case["chunks"]
    x = _beam_input(n * chunks, f, case["tsamp"], ranges, case["pulses"], seed)
    if case["where"] != "device":
        h = torch.empty(x.shape, dtype=torch.uint8, pin_memory=case["where"] == "pinned")
        h.copy_(x)
        x = h
    torch.cuda.synchronize()
    plan = dd.Plan(f, case["tsamp"], ranges, -(-n // 256) * 256, n_streams=case["streams"],
                   max_width=max(widths), peak_block=case["block"],
                   flags=dd.DD_FLAG_DEVICE_INPUT if case["where"] == "device" else 0)
    if case["search"] == "fused":
        plan.fuse_search(widths)
    parts = [x[n * k:n * (k + 1)] for k in range(chunks)]
    # deliver the stream's beginning: from here on every pass computes a full window
    while (plan.seq + 1) * n < plan.O or (plan.seq + 1) % chunks or plan.seq < 0:
        plan.run(parts[(plan.seq + 1) % chunks], n)
    plan.sync()
    return dict(case=case, plan=plan, parts=parts, ranges=ranges, widths=widths)


ROWS = 1 << 15  # candidate table of one chunk: its length follows the inputs, the table's does not


def _rows(v):
    out = np.zeros(ROWS, dtype=v.dtype)
    out[:v.size] = v
    return out


def _columns(c, t0):
    return dict(count=c.size, trial=_rows(c["trial"]), range=_rows(c["range"]),
                width=_rows(c["width"]), t_start=_rows(c["t_start"] - t0), snr=_rows(c["snr"]))


def run(state):
    case = state["case"]
    if case["kind"] == "static":
        y = state["y"]
        dd.dd_sps_static(y.data_ptr(), y.shape[0], y.shape[1], y.shape[1], 0, case["d"], 0,
                         state["widths"], case["threshold"], case["block"],
                         state["cands"].data_ptr(), state["cap"], state["count"].data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
        m = int(state["count"].item())  # the list's length; its order is left open
        raw = state["cands"][:m * dd.CAND_DTYPE.itemsize].cpu().numpy().view(dd.CAND_DTYPE)
        return _columns(raw[np.lexsort((raw["width"], raw["t_start"], raw["trial"]))], 0)
    if case["kind"] == "batch":
        b = state["batch"]
        b.run()
        b.wait()
        return [[_columns(b.candidates(k, j), 0) for j in range(b.info(k)[0])]
                for k in range(b.nbeams)]
    plan, n = state["plan"], case["n"]
    t0 = (plan.seq + 1) * n
    seqs = []
    for part in state["parts"]:
        seqs.append(plan.run(part, n))
        plan.search(state["widths"], case["threshold"],
                    estimator=dd.DD_EST_CLIPPED if case["search"] == "clipped" else None)
    out = dict(cands=[_columns(plan.candidates(s), t0) for s in seqs])
    if case["search"] != "fused":  # the last chunk's series, the plan's own buffers
        out["series"] = []
        for r, row in enumerate(state["ranges"]):
            ptr, m, stride, _ = dd.dd_series(plan.h, r)
            out["series"].append(_view(plan, ptr, (row[2], stride), "<i4")[:, :m])
    out["moments"] = []
    for r, row in enumerate(state["ranges"]):
        ptr, _ = dd.dd_moments(plan.h, r)
        out["moments"].append(_view(plan, ptr, (row[2], 4), "<i8")[:, :3])
    return out


# ---------------------------------------------------------------------------- work, exact


def work(case):
    """Input bytes read once and results written once; one add per channel and output sample."""
    if case["kind"] == "static":
        return {"bytes": 4.0 * case["trials"] * case["n"],
                "flops": 2.0 * case["trials"] * case["n"] * len(_ints(case["widths"]))}
    ranges = _ranges(case["ranges"])
    if case["kind"] == "batch":
        nbytes = flops = 0.0
        for c, n in zip(_ints(case["chans"]), _ints(case["lens"])):
            f = _freqs(c, 1550.0, 300.0) if c == 4096 else _freqs(c, 1450.0, 200.0)
            span = K_DM * 500.0 * (f.min() ** -2 - f.max() ** -2) / 64e-6
            nbytes += float(c) * n
            flops += sum(float(t) * ((n - span) // d) * c for _, _, t, d in ranges)
        return {"bytes": nbytes, "flops": flops}
    n = float(case["n"]) * case["chunks"]
    outs = sum(t * (n // d) for _, _, t, d in ranges)
    series = 0.0 if case["search"] == "fused" else 4.0 * outs
    return {"bytes": n * case["nchans"] + series, "flops": outs * case["nchans"]}


def _exact_search(y, widths, d, block, threshold, J0, t0, clipped):
    """Candidates of int64 series y [trials][n] with FP64 SNRs, as columns."""
    trials, n = y.shape
    nb = -(-n // block)
    P = torch.zeros((trials, n + 1), dtype=torch.int64, device=y.device)
    torch.cumsum(y, 1, out=P[:, 1:])
    yd = y.double()
    mean = yd.mean(1, keepdim=True)
    sd = (yd - mean).square().mean(1, keepdim=True).sqrt()
    best = torch.full((trials, nb), -math.inf, dtype=torch.float64, device=y.device)
    at = torch.zeros((trials, nb), dtype=torch.int64, device=y.device)
    wid = torch.zeros_like(at)
    for wo in widths:
        if wo < d or wo % d or wo // d > n:
            continue
        w = wo // d
        B = (P[:, w:] - P[:, :-w]).double()  # samples w - 1 .. n - 1
        if clipped:
            keep = torch.ones_like(B, dtype=torch.bool)
            for step in range(4):
                N = keep.sum(1, keepdim=True).double()
                mu = torch.where(keep, B, 0.0).sum(1, keepdim=True) / N
                dev = (torch.where(keep, B - mu, 0.0).square().sum(1, keepdim=True) / N).sqrt()
                if step < 3:
                    keep = (B >= torch.ceil(mu - 3.0 * dev)) & (B <= torch.floor(mu + 3.0 * dev))
            snr = (B - mu) / dev
        else:
            snr = (B - w * mean) / (math.sqrt(w) * sd)
        full = torch.full((trials, nb * block), -math.inf, dtype=torch.float64, device=y.device)
        full[:, w - 1:n] = snr
        v, i = full.view(trials, nb, block).max(2)
        j = i + block * torch.arange(nb, device=y.device)
        take = (v > best) | ((v == best) & (j < at))
        best, at = torch.where(take, v, best), torch.where(take, j, at)
        wid = torch.where(take, torch.full_like(wid, w), wid)
    tr, b = torch.nonzero(best >= float(np.float32(threshold)), as_tuple=True)
    j, w = at[tr, b], wid[tr, b]
    t = (J0 + j - w + 1) * d - t0
    snr = best[tr, b].cpu().numpy()
    key = np.lexsort(((w * d).cpu().numpy(), t.cpu().numpy(), tr.cpu().numpy()))
    return snr[key]


def _exact_series(x, freqs, tsamp, row, start, hi):
    """Series of one range in int64: x is the stream's uint8 window [samples][nchans] from global
    sample `start`; outputs the decimated samples from `start` to `hi`."""
    dm0, step, trials, d = row
    J = (hi - start) // d
    xd = x[:x.shape[0] // d * d].view(-1, d, x.shape[1]).sum(1, dtype=torch.int64).t().contiguous()
    dm = dm0 + np.arange(trials) * step
    a = 1.0 / (freqs * freqs) - 1.0 / (freqs.max() * freqs.max())
    s = np.floor((K_DM * dm)[:, None] * a[None, :] / (tsamp * d) + 0.5).astype(np.int64)
    y = torch.zeros((trials, J), dtype=torch.int64, device=x.device)
    for i in range(trials):
        for c in range(x.shape[1]):
            o = int(s[i, c])
            y[i] += xd[c, o:o + J]
    return y


def exact(case, seed):
    if case["kind"] == "static":
        if case["trials"] * case["n"] > 1.5e8:
            return None
        y = _series_input(case, seed).long()
        snr = _exact_search(y, _ints(case["widths"]), case["d"], case["block"],
                            case["threshold"], 0, 0, False)
        return dict(count=None, trial=None, range=None, width=None, t_start=None,
                    snr=_rows(snr))
    if case["kind"] != "beam":
        return None
    ranges, n = _ranges(case["ranges"]), case["n"]
    # one addition at a time from Python: the small beams only
    if case["chunks"] != 1 or case["nchans"] * sum(r[2] for r in ranges) > 4e5:
        return None
    f = _freqs(case["nchans"], case["fch1"], case["bw"])
    x = _beam_input(n, f, case["tsamp"], ranges, case["pulses"], seed)
    dmax = max(r[3] for r in ranges)
    a = f.min() ** -2 - f.max() ** -2
    need = 0
    for dm0, step, trials, d in ranges:
        tau = K_DM * (dm0 + (trials - 1) * step) * a
        need = max(need, d * int(math.floor(tau / (case["tsamp"] * d) + 0.5)))
    over = -(-need // dmax) * dmax
    if over > n:
        return None
    window = torch.cat([x[n - over:], x]) if over else x  # the same chunk came before
    out = []
    for r, row in enumerate(ranges):
        y = _exact_series(window, f, case["tsamp"], row, 0, n)
        out.append(_exact_search(y, _ints(case["widths"]), row[3], case["block"],
                                 case["threshold"], 0, over, case["search"] == "clipped"))
    none = [None] * len(ranges)
    got = dict(cands=[dict(count=None, trial=None, range=None, width=None, t_start=None,
                           snr=_rows(np.concatenate(out)))], moments=none)
    if case["search"] != "fused":
        got["series"] = none
    return got
