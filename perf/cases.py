"""Performance cases: what users of the selection have it do, through its public entry points.

A case is one call pattern on one kind of input.  The kinds of input are those of the repository's own
workloads: Poisson events (20 hits per layer in 10^3-event batches, 100 in batches of up to 10^6), log-normal
timeslices, dense six-station events, free-streaming timeslices.  They are drawn here on the GPU, because the
cases need fresh inputs often; the recipe (annulus 15 cm < r < 0.4 z, straight muons smeared by 0.1 cm, layers
10 cm apart) is that of the repository's generator.

Every output is a whole number (accept bits, counts, offsets, hit indices) and is defined bit by bit, so it is
compared for equality.  The order of triplet rows inside a unit is unspecified; a user who needs reproducible
rows sorts them, and so does ``run``.
"""
import math

import torch

import paper_1810_11966_gb300 as jp

DEV = "cuda"
PAPER_CUTS = (0.03, 0.025)  # cm^2, the paper's step 2b
LAYER_DZ, R_MIN, R_MAX_FRAC, SLOPE_MAX, SMEAR = 10.0, 15.0, 0.4, 0.35, 0.1
LN_MEDIAN, LN_SIGMA, COUNT_MIN, COUNT_MAX = 60.0, 1.0, 5, 1500
GAP_NS, JITTER_NS, WINDOW_NS, DT_NS = 100.0, 3.0, 100.0, 15.0


def _case(name=None, kind="run", events=1000, recipe="poisson", lam=100.0, stations=4, mode="chain", window=0.5,
          rows=False, z_table=False, distinct=False, p_two=0.01, p_one=0.05, slices=1):
    c = dict(kind=kind, events=events, recipe=recipe, lam=lam, stations=stations, mode=mode, window=window, rows=rows,
             z_table=z_table, distinct=distinct, p_two=p_two, p_one=p_one, slices=slices)
    return c if name is None else dict(c, name=name)


def listed():
    return [
        # an online node's smallest packet: 64 events, the trigger decision only; launches and host round trips count
        _case("run_64", events=64),
        # the 10^3-event workload (20 hits per layer, uniform in area, 30 % with two muons), trigger decision
        _case("run_1k", events=1000, recipe="uniform", lam=20.0, p_two=0.3, p_one=0.0),
        # the paper's own selection: trigger station only, printed cuts, its largest batch (8*10^4 events)
        _case("run_80k_paper", events=80_000, mode="paper", window=0.0),
        # the headline workload: 10^6 events in one call, triplets wanted
        _case("run_1m_rows", events=1_000_000, rows=True),
        # one log-normal timeslice of mean size: events of 5 to 1500 hits per layer side by side, trigger decision
        _case("slice_55k", events=55_000, recipe="lognormal"),
        # a small timeslice with the options on: triplets, hit-disjoint candidates, z from the detector geometry
        _case("slice_10k_options", events=10_000, recipe="lognormal", rows=True, distinct=True, z_table=True),
        # the dense stress shape: six stations, 1500 hits per layer, 1 cm window
        _case("dense_2k_6st", events=2_000, recipe="dense", lam=1500.0, stations=6, window=1.0, p_two=0.1, p_one=0.0),
        # a free-streaming timeslice of 10^5 collisions (windows built from hit times on the device)
        _case("stream_100k", kind="stream", events=100_000),
        # a short free-streaming timeslice, triplets wanted as indices into the timeslice
        _case("stream_1k_rows", kind="stream", events=1_000, rows=True),
        # events in pinned host memory, transfers inside the call, the paper's largest batch
        _case("host_80k", kind="host", events=80_000),
        # continuous batching: twelve timeslices in device memory over three slots, all submitted, all awaited
        _case("serve_12x10k", kind="serve", events=10_000, recipe="lognormal", slices=12),
        # the allocation-free counting call inside another program's event loop
        _case("noalloc_4k", kind="noalloc", events=4_000, lam=60.0),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: other sizes (odd ones among them), densities, windows, stations, options."""
    kind = rng.choice(["run"] * 6 + ["stream", "stream", "host", "serve", "serve", "noalloc"])
    paper = rng.random() < 0.25
    window = 0.0 if paper and rng.random() < 0.5 else round(_log_uniform(rng, 0.2, 1.0), 3)
    c = _case(kind=kind, mode="paper" if paper else "chain", window=window, p_two=0.01, p_one=0.05)
    if kind == "run":
        c["recipe"] = rng.choice(["poisson", "poisson", "uniform", "lognormal", "dense"])
        c["stations"] = rng.choice([1, 2, 3, 4, 4, 4, 4, 5, 6])
        c["z_table"] = rng.random() < 0.3
        c["distinct"] = rng.random() < 0.15
        if c["recipe"] == "dense":
            c["lam"] = round(_log_uniform(rng, 250.0, 1500.0), 1)
            c["events"] = int(_log_uniform(rng, 16, 1000))
        elif c["recipe"] == "lognormal":
            c["window"] = min(c["window"], 0.6)
            c["events"] = int(_log_uniform(rng, 1e3, 6e4))
            c["rows"] = rng.random() < 0.4
        else:
            c["lam"] = round(_log_uniform(rng, 5.0, 160.0), 1)
            cost = c["lam"] * c["stations"] * max(1.0, (c["window"] / 0.5) ** 2) * max(1.0, c["lam"] / 100.0)
            c["events"] = int(_log_uniform(rng, 64, min(1e6, 2e8 / cost)))
            c["rows"] = c["events"] <= 300_000 and rng.random() < 0.5
    elif kind == "stream":
        c["lam"] = round(_log_uniform(rng, 20.0, 110.0), 1)
        c["window"] = min(c["window"], 0.6)
        c["events"] = int(_log_uniform(rng, 300, 60_000))
        c["rows"] = c["events"] <= 900 and rng.random() < 0.5
    elif kind == "host":
        c["lam"] = round(_log_uniform(rng, 20.0, 110.0), 1)
        c["events"] = int(_log_uniform(rng, 500, 150_000))
        c["window"] = min(c["window"], 0.6)
    elif kind == "serve":
        c["recipe"], c["window"] = "lognormal", min(c["window"], 0.6)
        c["events"] = int(_log_uniform(rng, 1e3, 3e4))
        c["slices"] = rng.randint(3, 12)
    else:
        c["lam"] = round(_log_uniform(rng, 5.0, 70.0), 1)
        c["events"] = int(_log_uniform(rng, 64, 200_000))
    return c


# ------------------------------------------------------------------ inputs


def _layer_z(c):
    return [130.0 + 35.0 * s + d for s in range(c["stations"]) for d in (-LAYER_DZ, 0.0, LAYER_DZ)]


class _Recipe:
    """Signal content and hit counts of a batch of events, and the positions of any of its hits."""

    def __init__(self, c, seed):
        self.c, self.n, self.S3 = c, c["events"], 3 * c["stations"]
        self.g = torch.Generator(device=DEV).manual_seed(seed)
        u = self._u(self.n)
        self.n_mu = torch.where(u < c["p_two"], 2, torch.where(u < c["p_two"] + c["p_one"], 1, 0))
        self.slope = (2.0 * self._u(self.n, 2, 2) - 1.0) * SLOPE_MAX  # event, muon, plane
        if c["recipe"] == "lognormal":
            lam = LN_MEDIAN * torch.exp(LN_SIGMA * torch.randn(self.n, 1, generator=self.g, device=DEV))
            bg = torch.poisson(lam.clamp(COUNT_MIN, COUNT_MAX).expand(self.n, self.S3).contiguous(), generator=self.g)
            bg = bg.clamp(COUNT_MIN, COUNT_MAX)
        else:
            bg = torch.poisson(torch.full((self.n, self.S3), c["lam"], device=DEV), generator=self.g)
        self.counts = bg.long() + self.n_mu[:, None]
        # the muons' places in their layer: consecutive from a random one on
        self.first = (self._u(self.n, self.S3) * self.counts).long()
        self.z = torch.tensor(_layer_z(c), device=DEV)

    def _u(self, *shape):
        return torch.rand(*shape, generator=self.g, device=DEV)

    def positions(self, layer, local):
        """x, y, z of hit `local` of flat layer `layer` (event * 3S + layer of the detector)."""
        ev = layer // self.S3
        z = self.z[layer - ev * self.S3]
        if self.c["recipe"] == "uniform":
            r = torch.sqrt(R_MIN**2 + self._u(len(z)) * ((R_MAX_FRAC * z) ** 2 - R_MIN**2))
        else:
            r = R_MIN * torch.exp(self._u(len(z)) * torch.log(R_MAX_FRAC * z / R_MIN))
        phi = self._u(len(z)) * (2.0 * math.pi)
        x, y = r * torch.cos(phi), r * torch.sin(phi)
        cnt = self.counts.view(-1)[layer]
        rel = local - self.first.view(-1)[layer]
        rel = torch.where(rel < 0, rel + cnt, rel)
        at = (rel < self.n_mu[ev]).nonzero().squeeze(1)
        m = self.slope[ev[at], rel[at]]
        smear = SMEAR * torch.randn(len(at), 2, generator=self.g, device=DEV)
        x[at] = m[:, 0] * z[at] + smear[:, 0]
        y[at] = m[:, 1] * z[at] + smear[:, 1]
        return x, y, z


def _events(c, seed):
    """x, y, z and int32 offsets in the order event, station, layer."""
    r = _Recipe(c, seed)
    off = torch.zeros(r.n * r.S3 + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(r.counts.view(-1), 0, out=off[1:])
    step = max(1, int(3e7 / max(1.0, float(off[-1]) / r.n)))  # events at a time, for the size of the temporaries
    ends = off[:: step * r.S3].tolist() + [int(off[-1])]
    x, y, z = (torch.empty(ends[-1], device=DEV) for _ in range(3))
    for k, e0 in enumerate(range(0, r.n, step)):
        e1, h0 = min(r.n, e0 + step), ends[k]
        h1 = ends[k + 1] if e1 < r.n else ends[-1]
        layers = torch.arange(e0 * r.S3, e1 * r.S3, device=DEV)
        lay = torch.repeat_interleave(layers, r.counts[e0:e1].reshape(-1), output_size=h1 - h0)
        x[h0:h1], y[h0:h1], z[h0:h1] = r.positions(lay, torch.arange(h0, h1, device=DEV) - off[lay])
    return x, y, z, off.int(), int(r.counts.max()).bit_length()


def _timeslice(c, seed):
    """x, y, z, t, offsets of a free-streaming timeslice (groups of one layer, sorted by time) and its windows."""
    r = _Recipe(c, seed)
    # collisions at random times of a timeslice of fixed length (10^7 per second on average)
    when = torch.sort(torch.rand(r.n, generator=r.g, device=DEV, dtype=torch.float64))[0] * (GAP_NS * r.n)
    parts, off = [], [0]
    for q in range(r.S3):
        cnt = r.counts[:, q]
        ev = torch.repeat_interleave(torch.arange(r.n, device=DEV), cnt)
        local = torch.arange(len(ev), device=DEV) - (torch.cumsum(cnt, 0) - cnt)[ev]
        x, y, z = r.positions(ev * r.S3 + q, local)
        t = (when[ev] + JITTER_NS * torch.randn(len(ev), generator=r.g, device=DEV)).float()
        t, order = torch.sort(t)
        parts.append((x[order], y[order], z[order], t))
        off.append(off[-1] + len(ev))
    x, y, z, t = (torch.cat(p) for p in zip(*parts))
    bounds = torch.arange(int(GAP_NS * r.n / WINDOW_NS) + 1, device=DEV).float() * WINDOW_NS
    bits = max(b - a for a, b in zip(off, off[1:])).bit_length()
    return x, y, z, t, torch.tensor(off, dtype=torch.int32, device=DEV), bounds, bits


# ------------------------------------------------------------------ calls

_contexts = {}


def _params(c):
    t = PAPER_CUTS if c["window"] == 0.0 else (c["window"] ** 2,) * 2
    mode = jp.JPSI_MODE_PAPER if c["mode"] == "paper" else jp.JPSI_MODE_CHAIN
    return jp.params(c["stations"], mode, t_xz=t[0], t_yz=t[1], distinct_hits=int(c["distinct"]))


def _context(c):
    """The context that a process with these parameters keeps for all of its batches."""
    key = (c["kind"], c["stations"], c["mode"], c["window"], c["distinct"])
    if key not in _contexts:
        _contexts[key] = jp.Context(_params(c))
    return _contexts[key]


class _Outputs:
    """Output buffers of one batch of n events, and what they hold after a call."""

    def __init__(self, n, S, host=False):
        kw = dict(device="cpu", pin_memory=True) if host else dict(device=DEV)
        self.accept = torch.zeros((n + 31) // 32, dtype=torch.int32, **kw)
        self.tracks = torch.zeros(n, dtype=torch.int32, **kw)
        self.trip_off = torch.zeros(n * S + 1, dtype=torch.int64, **kw)
        self.rows = None
        o = self.o = jp.jpsi_outputs()
        o.accept_bits, o.track_counts = self.accept.data_ptr(), self.tracks.data_ptr()
        o.trip_off = self.trip_off.data_ptr()

    def want_rows(self, bits, room):
        """Room for the triplets: `room`, or what the counting call just made has found where that is more."""
        self.rows = torch.zeros((max(room, self.o.trip_needed), 3), dtype=torch.int32, device=DEV)
        self.o.triplets, self.o.trip_capacity = self.rows.data_ptr(), len(self.rows)
        self.place = torch.arange(len(self.rows), device=DEV)
        self.shift, self.weight = torch.tensor([2 * bits, bits, 0], device=DEV), 1 << 3 * bits

    def values(self):
        v = {"accept": self.accept, "tracks": self.tracks, "trip_off": self.trip_off}
        if self.rows is not None:
            # unit and three hit indices of each triplet in one integer, in a reproducible order; places past
            # the last triplet hold zeros and a unit past the last
            unit = torch.searchsorted(self.trip_off, self.place, right=True).sub_(1)
            key = torch.add((self.rows << self.shift).sum(1), unit, alpha=self.weight)
            v["rows"] = torch.sort(key)[0]
            self.rows.zero_()
        return v


def _rows_room(c):
    """Triplet rows that a user would allow for: signal, and background triplets as measured on the repository's
    workloads (they go with the cube of the hits per layer and the fourth power of the window's angle), and half as
    many again."""
    if c["recipe"] == "lognormal":  # mean of lambda^3, clipped
        u = [-5.0 + 0.01 * k for k in range(1001)]
        lam = [min(max(LN_MEDIAN * math.exp(LN_SIGMA * v), COUNT_MIN), COUNT_MAX) for v in u]
        cube = sum(a**3 * math.exp(-v * v / 2) for a, v in zip(lam, u)) * 0.01 / math.sqrt(2 * math.pi)
    else:
        cube = c["lam"] ** 3
    w = c["window"] or math.sqrt(max(PAPER_CUTS))
    zs = _layer_z(c)[1::3]
    rate = 700.0 if c["recipe"] == "uniform" else 2500.0
    per_event = sum(2 * c["p_two"] + c["p_one"] + rate * cube * (w / z) ** 4 for z in zs)
    return 2000 + int(1.5 * c["events"] * per_event)


def _check(status, ctx=None):
    if status != jp.JPSI_OK:
        raise jp.JpsiError(status, jp.jpsi_last_error(ctx) if ctx else "")


def _stream():
    return torch.cuda.current_stream().cuda_stream


def prepare(case, seed):
    c, S, n = case, case["stations"], case["events"]
    if c["kind"] == "serve":
        return _prepare_serve(c, seed)
    s = {"case": c, "kind": c["kind"]}
    if c["kind"] == "stream":
        x, y, z, t, off, bounds, bits = _timeslice(c, seed)
        s["hits"] = (x, y, z, t, off, bounds)
        s["in"] = jp.make_timeslice(x, y, z, t, off, bounds, DT_NS)
        n, call = len(bounds) - 1, jp.jpsi_run_stream
    else:
        x, y, z, off, bits = _events(c, seed)
        table = None
        if c["z_table"]:
            table, z = torch.tensor(_layer_z(c), device=DEV), None
        if c["kind"] == "host":
            x, y, z, off = (torch.empty_like(a, device="cpu", pin_memory=True).copy_(a) for a in (x, y, z, off))
        s["hits"] = (x, y, z, off, table)
        s["in"] = jp.make_batch(x, y, z, off, n, z_layer=table)
        call = jp.jpsi_run_host if c["kind"] == "host" else jp.jpsi_run
    if c["kind"] == "noalloc":
        s["params"] = _params(c)
        s["counts"] = [torch.zeros(m, dtype=torch.int32, device=DEV) for m in (n, n * S)]
    else:
        s["out"] = _Outputs(n, S, c["kind"] == "host")
        s["ctx"], s["call"] = _context(c), call
        if c["rows"]:
            torch.cuda.synchronize()
            _check(call(s["ctx"].ctx, s["in"], s["out"].o, _stream()), s["ctx"].ctx)
            s["out"].want_rows(bits, _rows_room(c))
    torch.cuda.synchronize()  # the inputs are there
    return s


def _prepare_serve(c, seed):
    batches, hits = [], []
    for k in range(c["slices"]):
        x, y, z, off, _ = _events(c, seed * 16 + k)
        hits.append((x, y, z, off))
        batches.append(jp.make_batch(x, y, z, off, c["events"]))
    outs = [_Outputs(c["events"], c["stations"]) for _ in batches]
    ctx = jp.Context(_params(c), hbm_budget=16 << 30)
    _check(jp.jpsi_serve_start(ctx.ctx, 3, c["events"], max(b.n_hits for b in batches), 0), ctx.ctx)
    torch.cuda.synchronize()
    return {"kind": "serve", "hits": hits, "batches": batches, "outs": outs, "ctx": ctx}


def run(state):
    s = state
    if s["kind"] == "serve":
        ctx, tickets = s["ctx"].ctx, []
        for b, o in zip(s["batches"], s["outs"]):
            status, ticket = jp.jpsi_serve_submit(ctx, b, o.o)
            _check(status, ctx)
            tickets.append(ticket)
        for ticket in tickets:
            status, result, _ = jp.jpsi_serve_wait(ctx, ticket)
            _check(status or result, ctx)
        return [o.values() for o in s["outs"]]
    if s["kind"] == "noalloc":
        tracks, units = s["counts"]
        _check(jp.jpsi_select_noalloc(s["params"], s["in"], tracks.data_ptr(), units.data_ptr(), _stream()))
        return {"tracks": tracks, "units": units}
    ctx = s["ctx"].ctx
    _check(s["call"](ctx, s["in"], s["out"].o, _stream()), ctx)
    return s["out"].values()


def work(case):
    """Bytes a pass cannot do without: the hits of the stations that the mode reads, the offsets and the outputs."""
    c, S, n = case, case["stations"], case["events"]
    lam = LN_MEDIAN * math.exp(LN_SIGMA**2 / 2) if c["recipe"] == "lognormal" else c["lam"]
    lam += 2 * c["p_two"] + c["p_one"]
    read = S if c["mode"] == "chain" else 1
    hits = n * 3 * read * lam
    per_hit = 16 if c["kind"] == "stream" else 8 if c["z_table"] else 12
    offsets = 4 * n * 3 * S if c["kind"] != "stream" else 4 * n
    out = 8 * n * S + 4 * n + n / 8 if c["kind"] != "noalloc" else 4 * n * S + 4 * n
    # three multiplications or divisions per hit for its slopes; the fits of the few candidates come on top
    return {"bytes": c["slices"] * (per_hit * hits + offsets + out), "flops": c["slices"] * 3.0 * hits}


def exact(case, seed):
    """All outputs are whole numbers: there is no value in 64 bits to hold them against."""
    return None
