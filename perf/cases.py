"""Performance cases: the work that users of this library have it do, through
its public entry points, on inputs shaped like the experiment's (6 x 9 = 54
crystals per calorimeter, 24 calorimeters, fills of up to 560,000 12-bit samples
at 800 MSPS).

A case is a dict of plain values:

  kind      fill    daq.process_fills on a device-resident batch
            batch   daq.BatchPlan (tuned, one graph launch) on a batch of uneven fills
            serve   daq.DaqServer: a burst of fills, drained
            host    daq.daq_process_fills_host: host buffers in, host buffers out
            xsum    daq.crystal_sum: per-crystal full-resolution fill sum
            pack    daq.pack_pool of the pool rows of a batch
            unpack  daq.unpack_pool of such a stream
  fills, calos, xtals, samples   the batch int16[fills][calos][xtals][samples]
  noise     per-crystal noise sigma (ADC counts); 3 marks ~94% of the samples,
            3 / sqrt(54) only those around pulses
  rate      pulses per calorimeter-fill, in units of the nominal 1,500
  uneven    fill lengths differ (device int32 fill_len), samples past a fill's
            length hold 4095
  threshold, pre, post, decim ("32", "8,32", ... or "")   the method's parameters
  sparse    DAQ_SPARSE (fill, serve)
  sync      fill, xsum: wait for the call and learn what it found; without it the
            call is queued, as in a loop over fills

Buffers come back whole, with what lies past the records, rows or bytes found
as prepare() left it.

Histograms are resident and accumulate from pass to pass, as in the DAQ.
"""
import math

import numpy as np
import torch

import paper_1611_04959_gb300 as daq

DEV = "cuda"
NOMINAL = 560_000             # samples of a 700 us fill
TAU = 64.4e3 / 1.25           # muon lifetime in samples
WIGGLE = 4365.0 / 1.25        # g-2 oscillation period in samples
QUIET = 108                   # no pulse before this sample
PULSE = 32                    # samples of a pulse that are generated


def _case(name, kind, calos, samples, fills=1, xtals=54, noise=3.0, rate=1.0, uneven=False, threshold=30, pre=8, post=24,
          decim="32", sparse=False, sync=False):
    c = dict(kind=kind, fills=fills, calos=calos, xtals=xtals, samples=samples, noise=noise, rate=rate, uneven=uneven,
             threshold=threshold, pre=pre, post=post, decim=decim, sparse=sparse, sync=sync)
    return dict(c, name=name) if name else c


QUIET_NOISE = round(3.0 / math.sqrt(54.0), 6)  # the 54-crystal sum has sigma ~3


def listed():
    return [
        # two calorimeters' first 25 us, waited for: monitoring, calibration runs, tests
        _case("fill_small", "fill", 2, 20_000, sync=True),
        # one calorimeter's whole fill, waited for: one frontend per calorimeter
        _case("fill_one_calo", "fill", 1, NOMINAL, sync=True),
        # the whole detector's fill in a loop over fills: the headline workload
        _case("fill_full", "fill", 24, NOMINAL),
        # the same with little noise: islands only around pulses, tiles without one passed over
        _case("fill_sparse", "fill", 24, NOMINAL, noise=QUIET_NOISE, sparse=True),
        # a short readout window whose row pitch is odd: rows share no alignment
        _case("fill_odd_pitch", "fill", 24, 100_003),
        # ten times the rate, low threshold, long tails kept, two histograms: the stress settings
        _case("fill_stress", "fill", 24, NOMINAL, fills=4, rate=10.0, threshold=15, post=64, decim="8,32"),
        # an accelerator cycle's fills of uneven length in one graph launch
        _case("batch_uneven", "batch", 24, NOMINAL, fills=6, uneven=True),
        # a burst of eight fills through the request loop, several in flight
        _case("serve_burst", "serve", 24, NOMINAL, fills=8),
        # a quarter of the detector from and to page-locked host memory
        _case("host_quarter", "host", 6, NOMINAL),
        # the whole detector's fill into the 5.8 GB per-crystal histograms
        _case("xsum_full", "xsum", 24, NOMINAL),
        # lossless packing of a whole fill's pool rows, and back
        _case("pack_full", "pack", 24, NOMINAL),
        _case("unpack_full", "unpack", 24, NOMINAL),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fill", "fill", "fill", "fill", "batch", "xsum", "pack", "unpack"])
    calos, samples = _log_int(rng, 1, 24), _log_int(rng, 4_000, NOMINAL)
    align = rng.random()
    if align < 0.6:
        samples = samples // 8 * 8
    elif align < 0.85:
        samples |= 1
    xtals = 54 if rng.random() < 0.7 else rng.choice([9, 25, 32, 33, 63, 64])
    fills = 1 if kind in ("pack", "unpack") else rng.choice([1, 1, 2, 3, 4])
    # at most the largest listed case's samples (three quarters of them for the
    # 16-byte histograms of xsum: one fill's worth)
    most = (1 if kind in ("xsum", "pack", "unpack") else 4) * 24 * 54 * NOMINAL
    while fills * calos * xtals * samples > most:
        fills, calos = max(1, fills - 1), max(1, calos - 1)
    sparse = rng.random() < 0.3
    post = rng.choice([24, 24, 16, 40, 64, 100])
    return _case(None, kind, calos, samples, fills, xtals, QUIET_NOISE if sparse else 3.0,
                 round(math.exp(rng.uniform(math.log(0.2), math.log(5.0))), 3), kind == "batch" or rng.random() < 0.25,
                 rng.choice([30, 30, 15, 50, 100]), rng.choice([8, 8, 0, 16]), post, rng.choice(["32", "32", "8,32", "16", "100"]),
                 sparse and kind == "fill", rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
def _decim(case):
    return tuple(int(d) for d in case["decim"].split(",") if d)


def _lens(case, seed):
    """Fill lengths, host: whole fills, or uniform between a seventh and the whole."""
    F, N = case["fills"], case["samples"]
    if not case["uneven"]:
        return [N] * F
    return [int(v) for v in np.random.default_rng([seed, 7]).integers(N // 7, N + 1, F)]


def _pulses(case, host, gen, length):
    """Fixed-point (1/1024 ADC) pulse heights of one calorimeter-fill: flat
    positions in [xtals][samples] and values.  Arrivals fall off with the muon
    lifetime and carry the g-2 oscillation; a pulse rises in 2 ns, decays with
    5 ns and spreads over the 3 x 3 crystals around its centre."""
    X, N = case["xtals"], case["samples"]
    n = int(host.poisson(1500 * case["rate"]))
    u = torch.rand(5, n, generator=gen, device=DEV, dtype=torch.float64)
    t = QUIET - TAU * torch.log1p(-u[0] * (1.0 - math.exp(-(NOMINAL - QUIET) / TAU)))
    keep = u[1] * 1.4 < 1.0 + 0.4 * torch.cos(2 * math.pi * t / WIGGLE)
    amp = 50.0 * torch.exp(u[2] * math.log(40.0)) * keep
    rows, cols = -(-X // 9), 9
    cr, cc = (u[3] * rows).long(), (u[4] * cols).long()
    d = torch.arange(-1, 2, device=DEV)
    r, c = cr[:, None, None] + d[:, None], cc[:, None, None] + d[None, :]
    x = r * cols + c
    inside = (r >= 0) & (r < rows) & (c >= 0) & (c < cols) & (x < X)
    w = torch.exp(-0.5 * (d[:, None] ** 2 + d[None, :] ** 2).double()) * inside
    w = w / w.sum(dim=(1, 2), keepdim=True).clamp_min(1e-9)
    k = t.floor().long()[:, None] + torch.arange(1, PULSE + 1, device=DEV)
    ns = (k - t[:, None]) * 1.25
    shape = torch.where(ns < 2.0, ns / 2.0, torch.exp(-(ns - 2.0) / 5.0)) * (k < length)
    v = (amp[:, None, None] * w.reshape(n, 9, 1) * shape[:, None, :] * 1024.0).round().int()
    at = x.reshape(n, 9, 1).clamp(0, X - 1) * N + k[:, None, :].clamp_max(N - 1)
    return at.reshape(-1), v.reshape(-1)


def _samples(case, seed):
    """int16[fills][calos][xtals][samples] on the device and the fill lengths."""
    F, C, X, N = case["fills"], case["calos"], case["xtals"], case["samples"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    host = np.random.default_rng(seed)
    lens = _lens(case, seed)
    out = torch.empty((F, C, X, N), dtype=torch.int16, device=DEV)
    ped = torch.randint(1700, 1901, (C, X, 1), generator=gen, device=DEV)
    noise = torch.empty((X, N), dtype=torch.float32, device=DEV)
    pulse = torch.empty((X, N), dtype=torch.int32, device=DEV)
    for f in range(F):
        for c in range(C):
            noise.normal_(0.0, case["noise"], generator=gen)
            at, v = _pulses(case, host, gen, lens[f])
            pulse.zero_().view(-1).index_add_(0, at, v)  # whole numbers: the same sum in any order
            noise.add_(pulse, alpha=1.0 / 1024.0).add_(ped[c]).round_().clamp_(0, 4095)
            out[f, c].copy_(noise)
        out[f, :, :, lens[f]:] = 4095
    return out, lens


def _pool_rows(case):
    """Rows packed: about what the method finds in such a batch."""
    return max(1, int(0.95 * _coverage(case) * _rows(case) * (4.0 / 7.0 if case["uneven"] else 1.0)))


def _rows(case):
    return case["fills"] * case["calos"] * case["samples"]


def _hdr_cap(case, fills=None):
    """Most islands: each is a window long at least, with a gap, but for those cut off at a fill's ends."""
    fc = (case["fills"] if fills is None else fills) * case["calos"]
    return fc * (case["samples"] // (case["pre"] + case["post"] + 2) + 2)


def _fit_rows(pool, rows):
    """The first `rows` pool rows; where fewer were found they come round again."""
    if len(pool) == 0:
        return torch.zeros((rows, pool.shape[1]), dtype=torch.int16, device=DEV)
    return torch.cat([pool] * -(-rows // len(pool)))[:rows].clone()


def _method(case):
    return dict(threshold=case["threshold"], pre=case["pre"], post=case["post"], decim=_decim(case))


def _outputs(case):
    o = daq.Outputs(torch, DEV, case["fills"], case["calos"], case["xtals"], _hdr_cap(case), _rows(case))
    o.hdr.zero_()
    o.pool.zero_()
    o.pedestal.zero_()
    return o


def _q(case):
    return torch.zeros(daq.q_size(case["calos"], case["samples"], _decim(case)), dtype=torch.int64, device=DEV)


def prepare(case, seed):
    C, X, N = case["calos"], case["xtals"], case["samples"]
    flags = daq.DAQ_SPARSE if case["sparse"] else 0
    x, lens = _samples(case, seed)
    fill_len = torch.tensor(lens, dtype=torch.int32, device=DEV) if case["uneven"] else None
    st = dict(case=case, x=x, fill_len=fill_len, flags=flags)
    kind = case["kind"]
    if kind in ("fill", "batch"):
        st.update(out=_outputs(case), q=_q(case))
    if kind == "fill":
        p = daq.make_params(fill_len=fill_len, flags=flags, **_method(case))
        st["ws"] = torch.empty(daq.daq_workspace_size(C, X, N, case["fills"], p), dtype=torch.uint8, device=DEV)
    elif kind == "batch":
        st["plan"] = daq.BatchPlan(x, st["q"], st["out"], fill_len=fill_len, flags=flags, **_method(case))
        torch.cuda.synchronize()
        # tuning leaves its own runs' results in the output buffers
        st["out"].hdr.zero_()
        st["out"].pool.zero_()
    elif kind == "serve":
        # worst-case slots are 1.6 GB each: room for the whole burst
        st["q"] = _q(case)
        st["server"] = daq.DaqServer(C, X, N, 14 << 30, auto_release=True, flags=flags, q=st["q"], max_slots=case["fills"],
                                     **_method(case))
        st["lens"] = lens
    elif kind == "host":
        host = torch.empty(x.shape, dtype=torch.int16, pin_memory=True)
        host.copy_(x)
        rows = _rows(case)
        out = daq.Outputs(torch, DEV, case["fills"], C, X, case["fills"] * C * ((N + 1) // 2), rows + 8 * 64)
        hdr = torch.zeros(_hdr_cap(case) * 3, dtype=torch.int64, pin_memory=True)
        pool = torch.zeros((rows, X), dtype=torch.int16, pin_memory=True)
        ped = torch.zeros((case["fills"], C, X), dtype=torch.int32, pin_memory=True)
        counts = torch.zeros(4, dtype=torch.int64, pin_memory=True)
        p = daq.make_params(fill_len=fill_len, flags=flags, stream=torch.cuda.current_stream(), **_method(case))
        ws = torch.empty(daq.daq_workspace_size(C, X, N, case["fills"], p), dtype=torch.uint8, device=DEV)
        p.workspace, p.workspace_bytes = ws.data_ptr(), ws.numel()
        io = daq.DaqHostIO(host.data_ptr(), x.data_ptr(), hdr.data_ptr(), hdr.numel() // 3, pool.data_ptr(), rows,
                           ped.data_ptr(), counts.data_ptr())
        st.update(host=host, out=out, hdr=hdr, pool=pool, ped=ped, counts=counts, p=p, ws=ws, io=io, q=_q(case))
    elif kind == "xsum":
        st["q"] = torch.zeros((C, X, N), dtype=torch.int64, device=DEV)
        st["ws"] = torch.empty(daq.daq_crystal_sum_workspace_size(C, X, case["fills"]), dtype=torch.uint8, device=DEV)
    else:
        res = daq.process_fills(x, fill_len=fill_len, hdr_cap=_hdr_cap(case), pool_cap=_rows(case), **_method(case))
        rows = _pool_rows(case)
        pool = _fit_rows(res["outputs"].pool[: res["n_rows"]], rows)
        st = dict(case=case, pool=pool, rows=rows)
        if kind == "pack":
            st["out"] = torch.zeros(daq.daq_pack_bound(rows, X), dtype=torch.uint8, device=DEV)
            st["ws"] = torch.empty(daq.daq_pack_workspace_size(rows, X), dtype=torch.uint8, device=DEV)
        else:
            st["packed"] = daq.pack_pool(pool, rows)[0].clone()
            del st["pool"]
    return st


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    C, X, N = case["calos"], case["xtals"], case["samples"]
    if kind == "fill":
        r = daq.process_fills(st["x"], fill_len=st["fill_len"], q=st["q"], outputs=st["out"], workspace=st["ws"],
                              flags=st["flags"], sync=case["sync"], **_method(case))
        o = r["outputs"]
        return dict(islands=o.hdr, pool=o.pool, pedestal=o.pedestal, counts=o.counts[:2], q=r["q"])
    if kind == "batch":
        st["plan"].launch(torch.cuda.current_stream())
        o = st["out"]
        return dict(islands=o.hdr, pool=o.pool, pedestal=o.pedestal, counts=o.counts[:2], q=st["q"])
    if kind == "serve":
        srv = st["server"]
        tickets = [srv.submit(st["x"][f], fill_len=st["lens"][f]) for f in range(case["fills"])]
        done = [srv.wait(t) for t in tickets]
        return dict(counts=np.array([[d["n_islands"], d["n_rows"]] for d in done], np.int64), q=st["q"])
    if kind == "host":
        rc = daq.daq_process_fills_host(C, X, N, case["fills"], st["p"], st["out"].struct(), st["q"].data_ptr(), st["io"])
        if rc != daq.DAQ_OK:
            raise daq.DaqError(rc, "daq_process_fills_host")
        return dict(islands=st["hdr"], pool=st["pool"], pedestal=st["ped"], counts=st["counts"][:2], q=st["q"])
    if kind == "xsum":
        return daq.crystal_sum(st["x"], q=st["q"], fill_len=st["fill_len"], workspace=st["ws"], sync=case["sync"])
    if kind == "pack":
        _, n = daq.pack_pool(st["pool"], st["rows"], out=st["out"], workspace=st["ws"])
        return dict(stream=st["out"], bytes=n)
    return daq.unpack_pool(st["packed"], st["rows"], X)


# ------------------------------------------------------------------ what a pass cannot do without
def _coverage(case):
    """Expected share of marked samples: a window holds a crossing of the noise, or a pulse does."""
    sigma = math.sqrt(case["xtals"] * (case["noise"] ** 2 + 1.0 / 12.0))
    p = 0.5 * math.erfc((case["threshold"] + 0.5) / sigma / math.sqrt(2.0))
    w = case["pre"] + case["post"] + 1
    t = np.linspace(0.0, case["samples"], 4096)
    lam = 1500.0 * case["rate"] / TAU * np.exp(-t / TAU)  # pulses per sample
    return float(np.mean(1.0 - (1.0 - p) ** w * np.exp(-lam * (w + 10))))


def work(case):
    # lengths depend on the seed only where fills are uneven: their mean there
    share = 4.0 / 7.0 if case["uneven"] else 1.0
    rows = _rows(case) * share
    cells = rows * case["xtals"]
    cover = _coverage(case)
    q = 16.0 * sum(case["calos"] * -(-case["samples"] // d) for d in _decim(case))
    adds = cells
    if case["kind"] == "xsum":
        return dict(bytes=2.0 * cells + 16.0 * case["calos"] * case["xtals"] * case["samples"], flops=2 * adds)
    if case["kind"] in ("pack", "unpack"):
        # the rows on one side, the stream on the other: a head word, and planes
        # for the spread of row to row differences, per crystal and 32 rows
        pool = 2.0 * case["xtals"] * _pool_rows(case)
        z = 2.0 * 2.7 * math.sqrt(2.0) * math.sqrt(case["noise"] ** 2 + 1.0 / 12.0)
        bits = 1.0 + math.ceil(math.log2(z))
        return dict(bytes=pool + pool / 16.0 * bits, flops=pool / 2.0)
    if case["kind"] == "serve":  # counts and histograms leave; the rows are written to the fill's slot
        return dict(bytes=2.0 * cells * (1.0 + cover) + q * case["fills"], flops=adds)
    return dict(bytes=2.0 * cells * (1.0 + cover) + q, flops=adds)


# ------------------------------------------------------------------ the same in plain torch, 64 bits
def _exact_fills(case, x, lens):
    F, C, X, N = x.shape
    decim = _decim(case)
    bins = [torch.zeros((C, -(-N // d)), dtype=torch.int64, device=DEV) for d in decim]
    peds, recs, pools, counts = [], [], [], []
    n_rows = 0
    for f in range(F):
        L, n = lens[f], min(100, lens[f])
        before = (sum(len(r) for r in recs), n_rows)
        for c in range(C):
            s = x[f, c, :, :L]
            ped = torch.div(s[:, :n].long().sum(1) + n // 2, max(n, 1), rounding_mode="floor")
            peds.append(ped.int())
            S = s.sum(0, dtype=torch.int64) - ped.sum()
            cross = torch.zeros(L + 1, dtype=torch.int64, device=DEV)
            cross[1:] = torch.cumsum(S > case["threshold"], 0)
            t = torch.arange(L, device=DEV)
            mark = cross[(t + case["pre"] + 1).clamp_max(L)] > cross[(t - case["post"]).clamp_min(0)]
            edge = torch.diff(torch.nn.functional.pad(mark.int(), (1, 1)))
            start, end = (edge == 1).nonzero()[:, 0], (edge == -1).nonzero()[:, 0]
            row = n_rows + torch.cumsum(end - start, 0) - (end - start)
            recs.append(torch.stack([torch.full_like(start, f | (c << 32)), start | ((end - start) << 32), row], 1))
            pools.append(s[:, mark].T.contiguous())
            n_rows += pools[-1].shape[0]
            for b, d in zip(bins, decim):
                k = -(-L // d)
                b[c, :k] += torch.nn.functional.pad(S, (0, k * d - L)).view(k, d).sum(1)
        counts.append((sum(len(r) for r in recs) - before[0], n_rows - before[1]))
    return dict(islands=torch.cat(recs).reshape(-1), pool=torch.cat(pools), pedestal=torch.stack(peds).view(F, C, X),
                counts=torch.tensor(counts, dtype=torch.int64), q=torch.cat([b.reshape(-1) for b in bins]))


def _exact_pack(pool):
    """The packed stream of pool rows, word by word (format: include/daq.h)."""
    rows, X = pool.shape
    nb = -(-rows // 32)
    if rows % 32:
        pool = torch.cat([pool, pool[-1:].expand(32 * nb - rows, X)])
    parts, sizes = [], []
    for b0 in range(0, nb, 1 << 15):
        v = pool[32 * b0: 32 * min(nb, b0 + (1 << 15))].view(-1, 32, X).long()
        d = torch.diff(v, dim=1, prepend=v[:, :1])
        z = torch.where(d >= 0, 2 * d, -2 * d - 1)
        top = z.amax(1)
        w = sum((top >> k > 0).long() for k in range(17))
        end = torch.cumsum((w + 1).reshape(-1), 0).view_as(w)
        at = end - (w + 1)
        words = torch.zeros(int(end[-1, -1]), dtype=torch.int64, device=DEV)
        words[at.reshape(-1)] = ((v[:, 0] & 0xFFFF) | (w << 16)).reshape(-1)
        bit = torch.arange(32, device=DEV)[None, :, None]
        for k in range(17):
            has = w > k
            words[(at + 1 + k)[has]] = (((z >> k) & 1) << bit).sum(1)[has]
        parts.append(words)
        sizes.append(4 * (w + 1).sum(1))
    offs = torch.zeros(nb + 1, dtype=torch.int64, device=DEV)
    if nb:
        offs[1:] = torch.cumsum(torch.cat(sizes), 0)
    words = torch.cat(parts) if parts else torch.zeros(0, dtype=torch.int64, device=DEV)
    words = torch.where(words >= 1 << 31, words - (1 << 32), words).int()
    head = torch.tensor([0x50514144 | (X << 32), rows], dtype=torch.int64, device=DEV)
    return torch.cat([head.view(torch.uint8), offs.view(torch.uint8), words.view(torch.uint8)])


def _whole(case, r):
    """The results at the front of the caller's whole buffers."""
    hdr = torch.zeros(_hdr_cap(case) * 3, dtype=torch.int64, device=DEV)
    hdr[: r["islands"].numel()] = r["islands"]
    pool = torch.zeros((_rows(case), case["xtals"]), dtype=torch.int16, device=DEV)
    pool[: len(r["pool"])] = r["pool"]
    return dict(r, islands=hdr, pool=pool)


def exact(case, seed):
    x, lens = _samples(case, seed)
    kind = case["kind"]
    if kind == "xsum":
        q = torch.zeros(x.shape[1:], dtype=torch.int64, device=DEV)
        for f, L in enumerate(lens):
            n = min(100, L)
            for c in range(x.shape[1]):
                ped = torch.div(x[f, c, :, :n].long().sum(1) + n // 2, max(n, 1), rounding_mode="floor")
                q[c, :, :L] += x[f, c, :, :L].long() - ped[:, None]
        return q
    r = _exact_fills(case, x, lens)
    if kind == "serve":
        return dict(counts=r["counts"], q=r["q"])
    r["counts"] = r["counts"].sum(0)
    if kind in ("pack", "unpack"):
        pool = _fit_rows(r["pool"], _pool_rows(case))
        if kind == "unpack":
            return pool
        stream = _exact_pack(pool)
        out = torch.zeros(daq.daq_pack_bound(*pool.shape), dtype=torch.uint8, device=DEV)
        out[: stream.numel()] = stream
        return dict(stream=out, bytes=stream.numel())
    return _whole(case, r)
