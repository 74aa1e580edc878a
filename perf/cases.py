"""Performance cases of the calorimeter hit path: the calls that programs make.

A program keeps one loaded geometry, one loaded parametrisation and a
workspace (``fcs.Simulator``) and calls it batch after batch; here the handle
is kept per case in the same way, so a call on new particles is what such a
program sees.  ``exact`` is the method in 64 bits in plain torch (Philox,
Poisson counts, inverse-CDF bins, cell lookup), sharing no code with the
library.
"""
import math

import numpy as np
import torch

from paper_2103_14737_gb300 import fcs, synth
from paper_2103_14737_gb300.autograd import simulate_cells

DEV = "cuda"


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
# sample: "electron" one 65.5 GeV electron per event, "ttbar" the hard scatter
# alone (400 particles), "pileup" the hard scatter plus Poisson(mu) collisions
# of 60 particles.  call: the entry point.  hit_E: the mean hit energies of
# the parametrisation ("std" 5-200 MeV; "fine" 0.5-20 MeV, ten times the hits).
def _case(name, call, sample, events, mu=0.0, mode="atomic", hit_E="std", interp=0):
    c = dict(call=call, sample=sample, events=events, mu=mu, mode=mode, hit_E=hit_E, interp=interp)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one electron, the paper's benchmark event: launches and latency
        _case("electron1", "simulate", "electron", 1),
        # an online trigger's call: one event, no device allocation
        _case("ttbar1_static", "static", "ttbar", 1),
        # the paper's single-electron sample in one batch: mostly empty cell rows
        _case("electrons500", "simulate", "electron", 500),
        # one hard-scatter event at fine hit energies (2.2M hits)
        _case("ttbar1_fine", "simulate", "ttbar", 1, hit_E="fine"),
        # a small odd batch with energy-bin interpolation
        _case("pileup7_interp", "simulate", "pileup", 7, mu=140.0, interp=1),
        # the ordinary production batch
        _case("pileup64", "simulate", "pileup", 64, mu=200.0),
        # the largest production batch (1.4e9 hits)
        _case("pileup1024", "simulate", "pileup", 1024, mu=200.0),
        # reproducible validation runs: small and ordinary batches
        _case("ttbar33_det", "simulate", "ttbar", 33, mode="det"),
        _case("pileup64_det", "simulate", "pileup", 64, mu=200.0, mode="det"),
        # a service that holds pinned host buffers (copies in and out included)
        _case("pileup64_host", "host", "pileup", 64, mu=200.0),
        # the adjoint of a production batch for a given dL/dE_cell
        _case("pileup64_backward", "backward", "pileup", 64, mu=200.0),
        # one fitting step: new tables, forward, loss, gradients (32 streams of one event)
        _case("ttbar32_train", "train", "ttbar", 32),
    ]


def draw(rng):
    def log_int(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))

    call = rng.choice(["simulate", "simulate", "simulate", "simulate", "static", "host", "backward", "train"])
    mode = "det" if call == "simulate" and rng.random() < 0.3 else "atomic"
    interp = 1 if call == "simulate" and rng.random() < 0.25 else 0
    sample = rng.choice(["electron", "ttbar", "pileup", "pileup"])
    mu = 0.0
    if call == "static":  # what the 16 MiB scratch holds
        sample = rng.choice(["electron", "ttbar"])
        events = rng.randint(1, 5)
    elif call == "train":
        sample = "ttbar"
        events = log_int(2, 64)
    elif sample == "pileup":
        mu = round(rng.uniform(20.0, 200.0), 1)
        events = log_int(1, 700 if call == "simulate" and mode == "atomic" else 100)
    else:
        events = log_int(1, 600)
    hit_E = "fine" if sample == "ttbar" and call != "train" and events <= 24 and rng.random() < 0.4 else "std"
    return _case(None, call, sample, events, mu, mode, hit_E, interp)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
HS = 400  # particles of a hard scatter


def _counts(case, seed):
    """Particles per event."""
    n = case["events"]
    if case["sample"] == "electron":
        return np.ones(n, dtype=np.int64)
    c = np.full(n, HS, dtype=np.int64)
    if case["sample"] == "pileup":
        rng = np.random.default_rng(seed)
        c += rng.poisson(60.0 * rng.poisson(case["mu"], size=n))
    return c


def _inputs(case, seed):
    """Particles on the device, and the random streams' seed and first event."""
    g = torch.Generator(DEV).manual_seed(1000003 * (seed + 1))
    cnt = torch.as_tensor(_counts(case, seed), device=DEV)
    off = torch.zeros(cnt.numel() + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(cnt, 0)
    n = int(off[-1])
    if case["sample"] == "electron":
        t = torch.zeros(n, dtype=torch.int32, device=DEV)
        E = torch.full((n,), 65536.0, device=DEV)
        eta = torch.full((n,), 0.22, device=DEV)
        phi = torch.zeros(n, device=DEV)
    else:
        if case["call"] == "train":  # the same event on every random stream
            n1, rep = HS, case["events"]
        else:
            n1, rep = n, 1

        def u():
            return torch.rand(n1, generator=g, device=DEV, dtype=torch.float64)

        first = torch.repeat_interleave(off[:-1], cnt)[:n1] if rep == 1 else torch.zeros(n1, dtype=torch.int64, device=DEV)
        k = torch.arange(n1, device=DEV) - first
        hard = k < HS
        uh = u()
        t_hard = torch.where(uh < 0.25, 0, torch.where(uh < 0.5, 1, 2))  # electrons, photons, charged pions
        t_mb = torch.where(uh < 0.1, 0, torch.where(uh < 0.4, 1, 2))
        t = torch.where(hard, t_hard, t_mb).int()
        E = (-torch.log1p(-u()) * torch.where(hard, 10000.0, 1500.0)).clamp(1000.0, 1.0e6).float()
        eta = ((2.0 * u() - 1.0) * torch.where(hard, 2.5, 3.2)).float()
        phi = ((2.0 * u() - 1.0) * math.pi).float()
        if rep > 1:
            t, E, eta, phi = (x.repeat(rep) for x in (t, E, eta, phi))
    return dict(type=t, E=E, eta=eta, phi=phi, event_offsets=off), 1 + 7919 * (seed % 100003), seed % 1000


_tables_kept = {}


def _tables(hit_E):
    """Geometry and parametrisation as host arrays (the program's files)."""
    if hit_E not in _tables_kept:
        geo = synth.geometry()
        _tables_kept[hit_E] = (geo, synth.params(geo, mean_hit_range=(5.0, 200.0) if hit_E == "std" else (0.5, 20.0)))
    return _tables_kept[hit_E]


_handle_kept = {}


def _handle(case):
    """The program's handle: loaded geometry, parametrisation and workspace."""
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _handle_kept:
        for sim in _handle_kept.values():
            sim.close()
        _handle_kept.clear()
        _handle_kept[key] = fcs.Simulator(*_tables(case["hit_E"]))
    return _handle_kept[key]


def _grad_rows(case, seed):
    geo, _ = _tables(case["hit_E"])
    g = torch.Generator(DEV).manual_seed(77003 * (seed + 1))
    return torch.randn((case["events"], geo.n_cells), generator=g, device=DEV)


def _train_tables(case, seed):
    """The tables of a fitting step: layer fractions within +-10 %, weights within +-20 % of the loaded ones."""
    _, prm = _tables(case["hit_E"])
    g = torch.Generator(DEV).manual_seed(31013 * (seed + 1))
    f = torch.as_tensor(prm.frac, device=DEV)
    w = torch.as_tensor(prm.shape_w, device=DEV)
    f = f * (0.9 + 0.2 * torch.rand(f.shape, generator=g, device=DEV))
    w = w * (0.8 + 0.4 * torch.rand(w.shape, generator=g, device=DEV))
    return f, w


def _train_target(case, seed):
    """Target energies (MeV): a fifth of the cells hit."""
    geo, _ = _tables(case["hit_E"])
    g = torch.Generator(DEV).manual_seed(52021 * (seed + 1))
    u = torch.rand((case["events"], geo.n_cells), generator=g, device=DEV)
    return torch.where(u < 0.2, -100.0 * torch.log(5.0 * u + 1e-6), torch.zeros((), device=DEV)).clamp_min(0.0)


def _capacity(case):
    """Entries of a program's output buffers: every cell of every event, at most 120M."""
    geo, _ = _tables(case["hit_E"])
    return min(case["events"] * geo.n_cells, 120_000_000)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.sim = case, _handle(case)
    s.parts, s.seed, s.first = _inputs(case, seed)
    if case["call"] in ("simulate", "static", "host"):
        # the program's own output buffers, zero beyond the cells that a call writes
        on = dict(device="cpu", pin_memory=True) if case["call"] == "host" else dict(device=DEV)
        s.out = dict(cell_ids=torch.zeros(_capacity(case), dtype=torch.int32, **on),
                     cell_E=torch.zeros(_capacity(case), dtype=torch.float32, **on),
                     event_offsets=torch.zeros(case["events"] + 1, dtype=torch.int64, **on))
    if case["call"] == "static":
        p = s.parts
        s.c_parts = fcs.fcs_particles(*(p[k].data_ptr() for k in ("type", "E", "eta", "phi", "event_offsets")))
    elif case["call"] == "host":
        s.batch = [s.parts[k].cpu().pin_memory().numpy() for k in ("type", "E", "eta", "phi", "event_offsets")]
        s.out_np = [s.out[k].numpy() for k in ("cell_ids", "cell_E", "event_offsets")]
        s.cfg = fcs.make_config()
        del s.parts
    elif case["call"] == "backward":
        s.g = _grad_rows(case, seed)
    elif case["call"] == "train":
        s.new_frac, s.new_w = _train_tables(case, seed)
        s.frac = torch.empty_like(s.new_frac).requires_grad_()
        s.w = torch.empty_like(s.new_w).requires_grad_()
        s.target = _train_target(case, seed)
    return s


def run(s):
    c, sim = s.case, s.sim
    if c["call"] == "simulate":
        mode = fcs.MODE_DETERMINISTIC if c["mode"] == "det" else fcs.MODE_ATOMIC
        sim.simulate(s.parts, s.seed, first_event=s.first, mode=mode, energy_interp=c["interp"], outputs=s.out)
        return s.out
    if c["call"] == "static":
        o = s.out
        fcs.fcs_simulate_events_static(sim.geo, sim.prm, s.c_parts, s.parts["E"].numel(), c["events"], s.seed, s.first,
                                       o["cell_ids"], o["cell_E"], o["event_offsets"])
        return o
    if c["call"] == "host":
        fcs.fcs_simulate_events_host(sim.geo, sim.prm, sim.ws, *s.batch, s.seed, s.first, s.cfg, *s.out_np)
        return s.out
    if c["call"] == "backward":
        g = sim.backward(s.parts, s.seed, s.g, first_event=s.first)
        return dict(d_frac=g["d_frac"], d_shape_w=g["d_shape_w"])
    # one fitting step: the optimiser has new values, written in place
    with torch.no_grad():
        s.frac.copy_(s.new_frac)
        s.w.copy_(s.new_w)
    s.frac.grad = s.w.grad = None
    cells = simulate_cells(sim, s.frac, s.w, s.parts, s.seed, s.first)
    loss = ((cells - s.target) ** 2).sum()
    loss.backward()
    return dict(cells=cells.detach(), loss=loss.detach(), d_frac=s.frac.grad, d_shape_w=s.w.grad)


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
# measured once per sample: hits and tasks per particle, non-zero cells per
# event at mu = 200 (they saturate slowly: taken as particles^0.75)
_HITS = {"electron": 1560.0, "ttbar": 553.0, "pileup": 94.0}
_TASKS = {"electron": 11.0, "ttbar": 8.3, "pileup": 6.8}
OPS_PER_HIT, OPS_PER_TASK = 117, 120  # arithmetic of the method, per pipe-independent operation


def work(case):
    n = case["events"]
    hs = n * (1 if case["sample"] == "electron" else HS)
    mb = n * 60.0 * case["mu"] if case["sample"] == "pileup" else 0.0
    kind = "electron" if case["sample"] == "electron" else "ttbar"
    hits = hs * _HITS[kind] + mb * _HITS["pileup"]
    if case["hit_E"] == "fine":
        hits *= 10.0
    tasks = hs * _TASKS[kind] + mb * _TASKS["pileup"]
    geo, prm = _tables(case["hit_E"])
    entries = prm.frac.size
    nnz = n * min(0.55 * geo.n_cells, 93000.0 * ((hs + mb) / n / 12400.0) ** 0.75)
    rows = min(float(entries), 400.0 if case["sample"] == "electron" else tasks)
    byts = 16.0 * (hs + mb) + 8.0 * (n + 1) + 520.0 * rows
    flops = OPS_PER_HIT * hits + OPS_PER_TASK * tasks
    if case["call"] == "backward":
        byts += 4.0 * n * geo.n_cells + 4.0 * entries * 129
    elif case["call"] == "train":  # tables in, gradients out, cells out and back
        byts += 2 * 4.0 * entries * 129 + 2 * 4.0 * n * geo.n_cells
        flops *= 2
    else:
        byts += 8.0 * nnz + 8.0 * (n + 1)
    return {"bytes": byts, "flops": float(flops)}


def tolerance(case):
    # atomic cells: one float product per group of hits and one rounding per
    # cell; deterministic cells are a fixed FP32 fold; gradients are sums of
    # FP32 products.  The cell ids and offsets are whole numbers and equal.
    if case["call"] in ("backward", "train"):
        return {"rel": 2e-7, "max": 1e-5}
    return {"rel": 2e-7, "max": 3e-6}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors (or integers) holding 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # 64-bit products; int64 wraps with the right bits
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return c0, c1, c2, c3


def _u53(a, b):
    return ((a >> 5).double() * 67108864.0 + (b >> 6).double()) * (1.0 / 9007199254740992.0)


def _poisson(mu, layer, particle, event, seed):
    n = torch.zeros_like(mu, dtype=torch.int64)
    ctr = layer | (1 << 16)
    i = ((mu < 10.0) & (mu > 0.0)).nonzero().squeeze(1)
    if i.numel():  # inversion by sequential search
        m = mu[i]
        x = _philox(torch.zeros_like(i), ctr[i], particle[i], event[i], seed)
        u = _u53(x[0], x[1])
        p = torch.exp(-m)
        F = p.clone()
        k = torch.zeros_like(i)
        j = 0
        go = u >= F
        while j < 200 and bool(go.any()):
            j += 1
            k = k + go
            p = p * m / j
            F = torch.where(go, F + p, F)
            go = go & (u >= F)
        n[i] = k
    i = (mu >= 10.0).nonzero().squeeze(1)
    if i.numel():  # PTRS (Hoermann 1993)
        n[i] = torch.floor(mu[i]).long()
        for it in range(64):
            if not i.numel():
                break
            m = mu[i]
            b = 0.931 + 2.53 * torch.sqrt(m)
            a = -0.059 + 0.02483 * b
            inv_alpha = 1.1239 + 1.1328 / (b - 3.4)
            vr = 0.9277 - 3.6224 / (b - 2.0)
            x = _philox(torch.full_like(i, it), ctr[i], particle[i], event[i], seed)
            U, V = _u53(x[0], x[1]) - 0.5, _u53(x[2], x[3])
            us = 0.5 - U.abs()
            kd = torch.floor((2.0 * a / us + b) * U + m + 0.43)
            quick = (us >= 0.07) & (V <= vr)
            drop = (kd < 0.0) | ((us < 0.013) & (V > us))
            lhs = torch.log(V) + torch.log(inv_alpha) - torch.log(a / (us * us) + b)
            rhs = -m + kd * torch.log(m) - torch.lgamma(kd.clamp_min(0.0) + 1.0)
            take = (us > 0.0) & (quick | (~drop & (lhs <= rhs)))
            n[i[take]] = kd[take].long()
            i = i[~take]
    return n


class _Exact64:
    """Tables of the method as FP64 device tensors."""

    def __init__(self, case, seed):
        geo, prm = _tables(case["hit_E"])
        self.geo, self.prm = geo, prm
        d = lambda a, t=torch.float64: torch.as_tensor(np.ascontiguousarray(a), device=DEV).to(t)  # noqa: E731
        if case["call"] == "train":
            f, w = _train_tables(case, seed)
            self.frac32, self.w = f.reshape(-1, geo.n_layers), w.reshape(-1, 128).double()
        else:
            self.frac32 = d(prm.frac, torch.float32).reshape(-1, geo.n_layers)
            self.w = d(prm.shape_w).reshape(-1, 128)
        self.mhe = d(prm.mean_hit_E).reshape(-1)
        C = torch.zeros_like(self.w)
        acc = torch.zeros_like(self.w[:, 0])
        for k in range(128):
            acc = acc + self.w[:, k]
            C[:, k] = acc
        thr = torch.floor(4294967296.0 * C / acc[:, None]).clamp_max(4294967295.0).long()
        ks = torch.arange(128, device=DEV)
        self.last = torch.where(self.w > 0.0, ks, -1).amax(1)
        self.thr = torch.where(ks < self.last[:, None], thr, torch.full_like(thr, 1 << 33)).reshape(-1)
        self.re, self.ae = d(prm.r_edges), d(prm.a_edges)
        r = geo.regions
        self.eta_lo, self.deta, self.phi_lo, self.dphi = (d(r[k]) for k in ("eta_lo", "deta", "phi_lo", "dphi"))
        self.ne, self.np_, self.co = (d(r[k], torch.int64) for k in ("n_eta", "n_phi", "cell_offset"))
        self.lrb = d(geo.layer_region_begin, torch.int64)
        split = np.full(len(r), -np.inf)
        for q in range(1, len(r)):
            if r["layer"][q] == r["layer"][q - 1]:
                split[q] = 0.5 * (r["eta_lo"][q - 1] + r["n_eta"][q - 1] * r["deta"][q - 1] + r["eta_lo"][q])
        self.split = d(split)
        self.max_regions = int(np.diff(geo.layer_region_begin).max())
        self.rz, self.barrel = d(geo.layers["rz"]), d(geo.layers["barrel"], torch.bool)

    def tasks(self, case, parts, seed, ev, pin):
        """(particle, layer, entry, float layer energy, hit count) of the particles' tasks."""
        NT, NE, NH, NL = self.prm.frac.shape
        E, eta = parts["E"].double(), parts["eta"].double()
        m, ex = torch.frexp(E)
        eb = ex.long() - 1 - self.prm.ebin_log2_min
        if case["interp"]:
            x = _philox(torch.zeros_like(pin), torch.full_like(pin, 2 << 16), pin, ev, seed)[0]
            eb = torch.where(x.double() / 4294967296.0 < 2.0 * m - 1.0, eb + 1, eb)
        eb = eb.clamp(0, NE - 1)
        hb = torch.floor(eta.abs() * self.prm.eta_bin_scale).long().clamp_max(NH - 1)
        row = (parts["type"].long() * NE + eb) * NH + hb
        El = (E[:, None] * self.frac32[row].double()).float()
        p, layer = (El > 0.0).nonzero(as_tuple=True)
        El = El[p, layer].double()
        entry = row[p] * NL + layer
        mu = (El / self.mhe[entry]).float().double()
        n = _poisson(mu, layer, pin[p], ev[p], seed).clamp_min(1)
        return p, layer, entry, El, n

    def hits(self, parts, seed, ev, pin, tasks):
        """(task, shape bin, cell) of every hit."""
        p, layer, entry, El, n = tasks
        t = torch.repeat_interleave(torch.arange(n.numel(), device=DEV), n)
        h = torch.arange(t.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[t]
        pt, lt = p[t], layer[t]
        x0, x1, x2, _ = _philox(h, lt, pin[pt], ev[pt], seed)
        base = entry[t] * 128
        lo, hi = torch.zeros_like(t), self.last[entry[t]]  # first k < last with x0 < T[k], else last
        for _ in range(7):
            mid = (lo + hi) >> 1
            right = (lo < hi) & (x0 >= self.thr[base + mid])
            hi = torch.where((lo < hi) & ~right, mid, hi)
            lo = torch.where(right, mid + 1, lo)
        b = lo
        del base, hi, mid, right, x0, h
        u24 = 1.0 / 16777216.0
        ir, ia = b >> 3, b & 7
        r = self.re[ir] + ((x1 >> 8).double() * u24) * (self.re[ir + 1] - self.re[ir])
        al = self.ae[ia] + ((x2 >> 8).double() * u24) * (self.ae[ia + 1] - self.ae[ia])
        del x1, x2, ir, ia
        # scale factors per task
        ec = parts["eta"].double()[p]
        R, bar = self.rz[layer], self.barrel[layer]
        sh = torch.sinh(ec.abs())
        mm = torch.tanh(ec.abs()) * sh / R
        s_phi = torch.where(bar, 1.0 / R, sh / R)
        s_eta = torch.where(bar, 1.0 / (R * torch.cosh(ec)), torch.where(ec < 0.0, mm, -mm))
        eta = ec[t] + r * torch.cos(al) * s_eta[t]
        phi = parts["phi"].double()[pt] + r * torch.sin(al) * s_phi[t]
        del r, al
        rb, end = self.lrb[lt], self.lrb[lt + 1]
        q = rb.clone()
        for k in range(1, self.max_regions):
            j = rb + k
            q = torch.where((j < end) & (eta >= self.split[j.clamp_max(len(self.split) - 1)]), j, q)
        ie = torch.floor((eta - self.eta_lo[q]) / self.deta[q]).clamp_min(0.0).long()
        ie = torch.minimum(ie, self.ne[q] - 1)
        ip = torch.remainder(torch.floor((phi - self.phi_lo[q]) / self.dphi[q]).long(), self.np_[q])
        return t, b, self.co[q] + ie * self.np_[q] + ip


def exact(case, seed):
    parts, sim_seed, first = _inputs(case, seed)
    X = _Exact64(case, seed)
    n_cells, off = X.geo.n_cells, parts["event_offsets"]
    grad = case["call"] in ("backward", "train")
    A = torch.zeros(X.w.numel(), dtype=torch.float64, device=DEV) if grad else None
    g_all = _grad_rows(case, seed) if case["call"] == "backward" else None
    target = _train_target(case, seed) if case["call"] == "train" else None
    cells, ids, vals, nz, loss = [], [], [], [0], 0.0
    lim = 100000 if case["hit_E"] == "fine" or case["sample"] != "pileup" else 250000
    if case["hit_E"] == "fine":
        lim //= 10
    h_off = off.cpu().numpy()
    e0 = 0
    while e0 < case["events"]:
        e1 = e0 + 1
        while e1 < case["events"] and e1 - e0 < 64 and (h_off[e1 + 1] - h_off[e0]) * (40 if case["sample"] == "electron" else 1) <= lim:
            e1 += 1
        a, b = int(h_off[e0]), int(h_off[e1])
        pt = {k: parts[k][a:b] for k in ("type", "E", "eta", "phi")}
        evl = torch.repeat_interleave(torch.arange(e0, e1, device=DEV), torch.diff(off[e0:e1 + 1]))
        pin = torch.arange(a, b, device=DEV) - off[evl]
        ev = evl + first
        tk = X.tasks(case, pt, sim_seed, ev, pin)
        t, bins, cell = X.hits(pt, sim_seed, ev, pin, tk)
        p, _, entry, El, n = tk
        Eh = (El / n).float().double()  # the method's float hit energy
        at = (evl[p][t] - e0) * n_cells + cell
        rows = torch.zeros((e1 - e0) * n_cells, dtype=torch.float64, device=DEV)
        if case["call"] != "backward":
            rows.index_add_(0, at, Eh[t])
        if grad:
            if case["call"] == "backward":
                g = g_all[e0:e1].reshape(-1).double()
            else:
                diff = rows - target[e0:e1].reshape(-1).double()
                g = 2.0 * diff
                loss = loss + (diff * diff).sum()
                cells.append(rows)
            A.index_add_(0, entry[t] * 128 + bins, Eh[t] * g[at])
        else:
            i = rows.nonzero().squeeze(1)
            ids.append((i % n_cells).int())
            vals.append(rows[i])
            nz += (nz[-1] + torch.cumsum(torch.bincount(i // n_cells, minlength=e1 - e0), 0)).tolist()
        del t, bins, cell, at, rows
        e0 = e1
    if not grad:
        pad = torch.zeros(_capacity(case) - nz[-1], dtype=torch.float64, device=DEV)
        return dict(cell_ids=torch.cat(ids + [pad.int()]), cell_E=torch.cat(vals + [pad]),
                    event_offsets=torch.tensor(nz, device=DEV))
    A = A.reshape(-1, 128)
    S, W, f = A.sum(1), X.w.sum(1), X.frac32.reshape(-1).double()
    hit = (A != 0.0).any(1)
    d_f = torch.where(hit & (f > 0.0), S / f, torch.zeros_like(S))
    d_w = torch.where(hit[:, None], torch.where(X.w > 0.0, A / X.w, torch.zeros_like(A)) - (S / W)[:, None], torch.zeros_like(A))
    if case["call"] == "backward":
        return dict(d_frac=d_f, d_shape_w=d_w.reshape(-1))
    shape = X.prm.frac.shape
    return dict(cells=torch.cat(cells).reshape(case["events"], n_cells), loss=loss, d_frac=d_f.reshape(shape),
                d_shape_w=d_w.reshape(X.prm.shape_w.shape))
