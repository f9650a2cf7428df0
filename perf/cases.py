"""The work that users of this framework have it do, as cases to be timed.

Each case goes through the package's public calls on a workload of the kind
the paper's pipeline runs (arXiv 2606.27262, Sec. 3: Band 3, 300-500 MHz,
1.31072 ms samples, up to 4096 channels, trial DMs up to 2000 pc cm^-3):
dedispersing one window, searching a DM transform, whole beams from device
and host memory, a batch of uneven beams, real-time gulps of several beams,
and the candidate classifier's scoring and its gradients.

Kinds (the "kind" of a case) and what they stand for:

* ``dmt``        stage one window and make its DM transform (a gulp, a
                 ragged block), integers out
* ``search``     boxcar search of a DM transform that is already on the GPU
* ``peaks``      the same with the (2r + 1)^2 peak window (11 x 11)
* ``map``        the best-S/N map, with any strictly increasing widths
* ``beam``       one beam resident on the GPU: dedispersion and search
* ``beam_host``  one beam from page-locked host memory, candidates back
* ``batch``      a step over beams of uneven length and DM range
* ``stream``     one gulp of each of several beams pushed and polled
* ``classify``   subband spectra -> two images -> probabilities
* ``peaks_cls``  a gulp's kept peaks: cut out of the staged window, imaged,
                 scored
* ``train``      loss and gradients of one training batch
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_2606_27262_gb300 as sp

TSAMP = 1.31072e-3
KDM = 4.148808e3
POW2 = [1, 2, 4, 8, 16, 32, 64, 128, 256]
MIXED = [1, 2, 3, 5, 8, 12, 20, 32, 50, 80]
FEAT = 256
CIN = (1, 16, 32, 64, 128)
COUT = (16, 32, 64, 128, 256)


# ------------------------------------------------------------------ cases --
def listed():
    return [
        # The smallest call in earnest: a 256-channel block from host memory,
        # where latency, launches and copies count.
        dict(name="small_beam_host", kind="beam_host", nchan=256, n_out=8192, dms="unit", max_dm=500, nw=6),
        # One 8 s gulp of one full-band beam, as a real-time loop makes it.
        dict(name="gulp_dmt", kind="dmt", nchan=4096, n_out=6104, dms="steps", max_dm=2000),
        # A block of ragged length from a 1024-channel mode, DM up to 500.
        dict(name="ragged_dmt", kind="dmt", nchan=1024, n_out=20011, dms="steps", max_dm=500),
        # The headline beam: 171.8 s of 4096 channels, 5751 trials, searched.
        dict(name="full_beam", kind="beam", nchan=4096, n_out=131072, dms="steps", max_dm=2000, nw=9),
        # The search alone, over every trial of a 43 s block.
        dict(name="search_block", kind="search", ndm=5751, n_out=32768, nchan=4096, nw=9),
        # Best-S/N map with widths that are not powers of two, odd length
        # (diagnostic plots of one DM range).
        dict(name="map_mixed_widths", kind="map", ndm=501, n_out=20011, nchan=4096, nw=10),
        # The 11 x 11 stencil of the paper's peak filter.
        dict(name="peaks_11x11", kind="peaks", ndm=1751, n_out=16384, nchan=4096, nw=9, radius=5),
        # Uneven beams in one step (the multi-beam workload of one GPU).
        dict(name="uneven_batch", kind="batch", nchan=4096, n_outs="16384,20483,40000", max_dms="500,2000,1000", nw=9),
        # Six beams' gulps arriving together at the streaming search.
        dict(name="stream_gulps", kind="stream", nchan=4096, beams=6, n_out=6104, dms="steps", max_dm=2000, nw=9),
        # Scoring a large batch of candidates.
        dict(name="classify_batch", kind="classify", batch=256, t_in=512),
        # Scoring the few kept peaks of one gulp.
        dict(name="gulp_peaks", kind="peaks_cls", nchan=4096, n_out=6104, dms="steps", max_dm=2000, ncand=5, t_in=512),
        # Gradients of one training batch.
        dict(name="train_batch", kind="train", batch=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dmt", "dmt", "dmt", "beam", "beam", "beam_host", "search", "search", "peaks", "map", "batch",
                       "stream", "classify", "peaks_cls", "train"])
    nw = rng.randint(5, 9)
    if kind in ("dmt", "beam"):
        nchan = rng.choice([256, 512, 1000, 1024, 2048, 4096, 4096])
        dms = rng.choice(["steps", "steps", "steps", "unit"])
        max_dm = rng.randint(100, 500) if dms == "unit" else rng.randint(100, 2000)
        c = dict(kind=kind, nchan=nchan, n_out=_log(rng, 4096, 131072 if kind == "beam" else 40000), dms=dms,
                 max_dm=max_dm)
        return dict(c, nw=nw) if kind == "beam" else c
    if kind == "beam_host":
        return dict(kind=kind, nchan=rng.choice([256, 512]), n_out=_log(rng, 4096, 32768), dms="unit",
                    max_dm=rng.randint(100, 500), nw=nw)
    if kind in ("search", "peaks", "map"):
        big = kind == "search"
        c = dict(kind=kind, ndm=_log(rng, 200, 5751 if big else 2000), n_out=_log(rng, 6000, 65536 if big else 24000),
                 nchan=rng.choice([256, 1024, 4096]), nw=nw)
        return dict(c, radius=rng.randint(2, 5)) if kind == "peaks" else c
    if kind == "batch":
        n = rng.randint(2, 4)
        return dict(kind=kind, nchan=rng.choice([1024, 4096]), nw=nw,
                    n_outs=",".join(str(_log(rng, 8192, 32768)) for _ in range(n)),
                    max_dms=",".join(str(rng.choice([500, 1000, 2000])) for _ in range(n)))
    if kind == "stream":
        return dict(kind=kind, nchan=rng.choice([1024, 4096]), beams=rng.randint(2, 6), n_out=rng.randint(4000, 8000),
                    dms="steps", max_dm=rng.randint(200, 2000), nw=nw)
    if kind == "classify":
        return dict(kind=kind, batch=_log(rng, 4, 256), t_in=rng.choice([512, 512, 400]))
    if kind == "peaks_cls":
        return dict(kind=kind, nchan=rng.choice([1024, 4096]), n_out=rng.randint(4000, 8000), dms="steps",
                    max_dm=rng.randint(200, 2000), ncand=rng.randint(1, 64), t_in=512)
    return dict(kind=kind, batch=_log(rng, 8, 96))


# ------------------------------------------------------------ axes, plans --
def freqs(nchan):
    return 500.0 - np.arange(nchan, dtype=np.float64) * (200.0 / nchan)


def trial_dms(dms, max_dm):
    """"unit": 0..max_dm in steps of 1; "steps": the paper's schedule of
    0.1 / 0.2 / 0.5 / 1.0 over [0, 250) / [250, 500) / [500, 1000) /
    [1000, 2000), then 2000, cut at max_dm."""
    if dms == "unit":
        return np.arange(0, max_dm + 1, dtype=np.float64)
    parts = [lo + step * np.arange(int(round((hi - lo) / step)), dtype=np.float64)
             for lo, hi, step in ((0.0, 250.0, 0.1), (250.0, 500.0, 0.2), (500.0, 1000.0, 0.5), (1000.0, 2000.0, 1.0))]
    v = np.concatenate(parts + [np.array([2000.0])])
    return v[v <= max_dm + 1e-9]


@functools.lru_cache(maxsize=None)
def plan_of(nchan, dms, max_dm):
    """A program makes its band's plan once and keeps it."""
    return sp.Plan(freqs(nchan), TSAMP, trial_dms(dms, max_dm))


def max_delay(nchan, dms, max_dm):
    f = freqs(nchan)
    dm = float(trial_dms(dms, max_dm)[-1])
    return int(np.floor(KDM * dm * (1.0 / (f[-1] * f[-1]) - 1.0 / (f[0] * f[0])) / TSAMP + 0.5))


# ----------------------------------------------------------------- inputs --
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + salt)
    return g


def make_beam(seed, nchan, n_in, n_out, max_dm, salt=0, wrap=0):
    """8-bit filterbank [n_in][nchan] on the GPU: N(128, 16) with a gentle
    bandpass, dispersed bursts, a few narrowband channels and a broadband
    impulse.  wrap > 0: the first `wrap` samples repeat periodically."""
    gen = _gen(seed, salt)
    rng = np.random.default_rng((int(seed), salt, nchan))
    rows = wrap or n_in
    x = torch.empty((rows, nchan), dtype=torch.uint8, device="cuda")
    gain = (16.0 * (0.8 + 0.4 * torch.rand(nchan, generator=gen, device="cuda")))
    for r in range(0, rows, 16384):
        n = min(16384, rows - r)
        v = torch.randn((n, nchan), generator=gen, device="cuda", dtype=torch.float32).mul_(gain).add_(128.0)
        x[r:r + n] = v.round_().clamp_(0, 255).to(torch.uint8)
    f = freqs(nchan)
    ch = torch.arange(nchan, device="cuda")
    for _ in range(max(2, min(20, n_out // 6000))):
        dm, w = rng.uniform(0.05, 0.95) * max_dm, int(rng.integers(1, 12))
        t0 = int(rng.integers(64, max(65, n_out - 128)))
        amp = 16.0 * rng.uniform(9.0, 20.0) / math.sqrt(nchan * w)
        d = torch.as_tensor(np.round(KDM * dm * (1.0 / (f * f) - 1.0 / (f[0] * f[0])) / TSAMP).astype(np.int64),
                            device="cuda")
        t = (t0 + d)[:, None] + torch.arange(w, device="cuda")[None, :]
        if wrap:
            t = t % rows
        add = (amp + torch.rand(t.shape, generator=gen, device="cuda")).floor_()
        ok = t < rows
        tt, cc = t[ok], ch[:, None].expand_as(t)[ok]
        x[tt, cc] = (x[tt, cc].float() + add[ok]).clamp_(0, 255).to(torch.uint8)
    for c in rng.integers(0, nchan, size=3):
        x[:, int(c)] = (x[:, int(c)].float() + 30.0).clamp_(0, 255).to(torch.uint8)
    r = int(rng.integers(0, rows))
    x[r] = (x[r].float() + 1.0).clamp_(0, 255).to(torch.uint8)
    if wrap:
        x = x.repeat((n_in + rows - 1) // rows, 1)[:n_in].contiguous()
    return x


def make_dmt(seed, ndm, n_out, nchan):
    """A DM transform [ndm][n_out]: noise about 128 nchan with the channel
    sum's deviation, a slow drift, and pulses that widen and fade with the
    distance from their trial DM."""
    gen = _gen(seed, 7)
    sig = 16.0 * math.sqrt(nchan)
    x = torch.empty((ndm, n_out), dtype=torch.int32, device="cuda")
    drift = torch.sin(torch.arange(n_out, device="cuda") * (2.0 * math.pi / 30000.0)) * (0.03 * sig)
    for r in range(0, ndm, 512):
        n = min(512, ndm - r)
        v = torch.randn((n, n_out), generator=gen, device="cuda", dtype=torch.float32).mul_(sig)
        x[r:r + n] = v.add_(drift).add_(128.0 * nchan).round_().clamp_(0, 255.0 * nchan).to(torch.int32)
    rng = np.random.default_rng((int(seed), ndm, 11))
    for _ in range(max(4, min(40, n_out // 1000))):
        d0, t0, w = int(rng.integers(0, ndm)), int(rng.integers(8, n_out - 400)), int(rng.integers(1, 64))
        total = sig * math.sqrt(w) * rng.uniform(9.0, 30.0)
        dd = np.arange(max(0, d0 - 40), min(ndm, d0 + 41))
        ww = w + np.abs(dd - d0) // 2
        rr = np.repeat(dd, ww)
        cc = t0 + np.concatenate([np.arange(k) for k in ww])
        vv = np.repeat(np.round(total / ww), ww)
        at = (torch.as_tensor(rr, device="cuda"), torch.as_tensor(cc, device="cuda"))
        x.index_put_(at, torch.as_tensor(vv.astype(np.int32), device="cuda"), accumulate=True)
    return x


def make_spectra(seed, batch, t_in):
    """Subband dynamic spectra [batch][256][t_in]: unit noise, half of them
    with a pulse near the centre, a quarter with narrowband lines."""
    gen = _gen(seed, 13)
    x = torch.randn((batch, 256, t_in), generator=gen, device="cuda", dtype=torch.float32)
    rng = np.random.default_rng((int(seed), batch, 17))
    u = torch.arange(t_in, device="cuda", dtype=torch.float32)
    s = torch.arange(256, device="cuda", dtype=torch.float32)[:, None] / 255.0
    for q in range(batch):
        if q % 2 == 0:
            c = t_in / 2 + rng.uniform(-2, 2) + rng.uniform(-12, 12) * s
            w = rng.uniform(1.0, 8.0)
            x[q] += rng.uniform(0.5, 2.5) * torch.exp(-0.5 * ((u[None, :] - c) / w) ** 2)
        elif q % 4 == 1:
            x[q, torch.as_tensor(rng.integers(0, 256, size=6), device="cuda")] += 4.0
    return x


def make_params(seed):
    """Weights as a network in use has them: He-scaled, small biases."""
    rng = np.random.default_rng((int(seed), 19))
    parts = []
    for _ in range(2):
        for ci, co in zip(CIN, COUT):
            parts.append(rng.standard_normal(co * 9 * ci) * math.sqrt(2.0 / (9 * ci)))
            parts.append(rng.standard_normal(co) * 0.05)
        parts.append(rng.standard_normal(FEAT) * math.sqrt(1.0 / FEAT))
        parts.append(np.zeros(1))
    return np.concatenate(parts).astype(np.float32)


def make_images(seed, batch):
    """Standardised bf16 image pairs and labels of a training batch."""
    gen = _gen(seed, 23)
    out = []
    for _ in range(2):
        x = torch.randn((batch, 256, 256), generator=gen, device="cuda", dtype=torch.float32)
        x[::2, :, 124:132] += 1.0
        x -= x.mean(dim=(1, 2), keepdim=True)
        x /= x.std(dim=(1, 2), keepdim=True)
        out.append(x.to(torch.bfloat16))
    labels = torch.zeros(batch, dtype=torch.float32, device="cuda")
    labels[::2] = 1.0
    return out[0], out[1], labels


def _bytes(n):
    return torch.empty(max(int(n), 16), dtype=torch.uint8, device="cuda")


def _widths(case):
    w = MIXED if case["kind"] == "map" else POW2
    return np.array(w[:case["nw"]], dtype=np.int32)


def _cand_cap(case):
    """Room for every candidate the inputs give, as a program leaves it."""
    return {"beam": 1 << 17, "beam_host": 1 << 13, "stream": 1 << 14, "search": 1 << 16}.get(case["kind"], 1 << 15)


# ---------------------------------------------------------------- prepare --
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dmt", "beam", "beam_host"):
        plan = plan_of(case["nchan"], case["dms"], case["max_dm"])
        n_in = case["n_out"] + plan.max_delay
        x = make_beam(seed, case["nchan"], n_in, case["n_out"], case["max_dm"])
        if kind == "dmt":
            return dict(kind=kind, plan=plan, x=x, work=_bytes(sp.dedisperse_workspace_bytes(plan, n_in)),
                        out=torch.empty((plan.ndm, case["n_out"]), dtype=torch.int32, device="cuda"))
        cap = _cand_cap(case)
        s = sp.Searcher(plan, case["n_out"], _widths(case), 6.0, 8192, cap)
        if kind == "beam":
            return dict(kind=kind, s=s, x=x, cands=torch.zeros((cap, 4), dtype=torch.int32, device="cuda"),
                        count=torch.zeros(1, dtype=torch.int64, device="cuda"))
        return dict(kind=kind, s=s, x=x.cpu().pin_memory(), cands=np.zeros((cap, 4), np.int32))
    if kind in ("search", "peaks", "map"):
        w = _widths(case)
        x = make_dmt(seed, case["ndm"], case["n_out"], case["nchan"])
        st = dict(kind=kind, x=x, w=w, work=_bytes(sp.sps_workspace_bytes(case["ndm"], case["n_out"], w.size, 8192)))
        if kind == "map":
            st.update(best=torch.empty(x.shape, dtype=torch.float32, device="cuda"),
                      wbest=torch.empty(x.shape, dtype=torch.int8, device="cuda"))
            return st
        if kind == "peaks":
            st.update(radius=case["radius"], work=_bytes(sp.sps_window_workspace_bytes(
                case["ndm"], case["n_out"], w.size, 8192, case["radius"])))
        st.update(cands=torch.zeros((_cand_cap(case), 4), dtype=torch.int32, device="cuda"),
                  count=torch.zeros(1, dtype=torch.int64, device="cuda"))
        return st
    if kind == "batch":
        n_outs, max_dms = _ints(case["n_outs"]), _ints(case["max_dms"])
        uniq = sorted(set(max_dms))
        plans = [plan_of(case["nchan"], "steps", m) for m in uniq]
        b = sp.Batch(plans, [uniq.index(m) for m in max_dms], n_outs, _widths(case), 6.0, 8192, _cand_cap(case), 4 << 30)
        for i, (n, m) in enumerate(zip(n_outs, max_dms)):
            dst = b.input_tensor(i, case["nchan"])
            dst.copy_(make_beam(seed, case["nchan"], int(dst.shape[0]), n, m, salt=i))
        return dict(kind=kind, b=b)
    if kind == "stream":
        plan = plan_of(case["nchan"], case["dms"], case["max_dm"])
        gulp, row = case["n_out"], case["nchan"]
        # Rings, and slots for a batch in flight and one being collected.
        slot = 2 * (gulp + plan.max_delay + 640) * row + plan.ndm * gulp * 5 + (64 << 20)
        st = sp.Stream(plan, case["beams"], gulp, _widths(case), 6.0, 8192, _cand_cap(case),
                       case["beams"] * ((gulp + plan.max_delay) * row + 3 * slot) + (1 << 30), max_batch=16)
        gulps = []
        for b in range(case["beams"]):
            # The sky repeats with the gulp, so that every pass sees the same windows.
            x = make_beam(seed, row, gulp, gulp, case["max_dm"], salt=b, wrap=gulp).cpu()
            L = plan.max_delay
            reps = (L + gulp - 1) // gulp
            h = x.repeat(max(reps, 1), 1)
            st.history(b, h[h.shape[0] - L:].contiguous() if L else h[:1].contiguous())
            gulps.append(x.pin_memory())
        return dict(kind=kind, st=st, gulps=gulps)
    if kind in ("classify", "peaks_cls"):
        clf = sp.Classifier(max_batch=256 if kind == "classify" else 64, seed=0)
        clf.set_params(make_params(seed))
        t_in = case["t_in"]
        B = case["batch"] if kind == "classify" else case["ncand"]
        shift = torch.as_tensor(sp.dmt_shifts(freqs(4096), 256, (t_in - 256) // 2), device="cuda")
        img = [torch.empty((B, 256, 256), dtype=torch.bfloat16, device="cuda") for _ in range(2)]
        st = dict(kind=kind, clf=clf, shift=shift, ft=img[0], dmt=img[1],
                  work=_bytes(sp.library().sp_cnn_features_workspace_bytes(B)),
                  prob=torch.empty(B, dtype=torch.float32, device="cuda"), t_in=t_in)
        if kind == "classify":
            st["sub"] = make_spectra(seed, B, t_in)
            return st
        plan = plan_of(case["nchan"], case["dms"], case["max_dm"])
        n_in = case["n_out"] + plan.max_delay
        x = make_beam(seed, case["nchan"], n_in, case["n_out"], case["max_dm"])
        staged = sp.staged_buffer(case["nchan"], n_in)
        sp.stage_input(x, staged)
        st.update(plan=plan, staged=staged, n_in=n_in, cands=torch.as_tensor(_peaks(case, plan.ndm, seed), device="cuda"))
        return st
    clf = sp.Classifier(max_batch=96, seed=0)
    clf.set_params(make_params(seed))
    ft, dmt, labels = make_images(seed, case["batch"])
    return dict(kind=kind, clf=clf, ft=ft, dmt=dmt, labels=labels)


def _ints(text):
    return [int(v) for v in str(text).split(",")]


def _peaks(case, ndm, seed):
    """Kept peaks of a gulp: (trial, sample, width index, S/N bits)."""
    rng = np.random.default_rng((int(seed), case["ncand"], 29))
    n = case["ncand"]
    c = np.zeros((n, 4), np.int32)
    c[:, 0] = np.sort(rng.integers(ndm // 20, ndm, size=n))
    c[:, 1] = rng.integers(0, case["n_out"] - 256, size=n)
    c[:, 2] = rng.integers(0, 6, size=n)
    c[:, 3] = rng.uniform(10, 30, size=n).astype(np.float32).view(np.int32)
    return c


# -------------------------------------------------------------------- run --
def _on_gpu(cands, count):
    """The found candidates in (trial, sample) order at the head of a list of
    the program's own capacity, left on the GPU; the program reads the count
    to know how many there are."""
    n = min(int(count.item()), cands.shape[0])
    c = cands[:n]
    where = torch.full((cands.shape[0], 3), -1, dtype=torch.int32, device=cands.device)
    snr = torch.zeros(cands.shape[0], dtype=torch.float32, device=cands.device)
    c = c[torch.argsort((c[:, 0].to(torch.int64) << 32) | c[:, 1].to(torch.int64))]
    where[:n] = c[:, :3]
    snr[:n] = c[:, 3].contiguous().view(torch.float32)
    return {"count": count, "where": where, "snr": snr}


def _on_host(c, cap, n):
    where, snr = np.full((cap, 3), -1, np.int32), np.zeros(cap, np.float32)
    c = c[np.lexsort((c[:, 1], c[:, 0]))]
    where[:c.shape[0]] = c[:, :3]
    snr[:c.shape[0]] = np.ascontiguousarray(c[:, 3]).view(np.float32)
    return {"count": n, "where": where, "snr": snr}


def _records(rec, cap):
    """The same from the package's sorted candidate records."""
    return _on_host(np.ascontiguousarray(rec).view(np.int32).reshape(-1, 4), cap, int(rec.size))


def run(state):
    kind = state["kind"]
    if kind == "dmt":
        sp.dedisperse(state["plan"], state["x"], state["out"], state["work"])
        return state["out"]
    if kind == "beam":
        state["s"].run(state["x"], state["cands"], state["count"])
        return _on_gpu(state["cands"], state["count"])
    if kind == "beam_host":
        n = state["s"].run_host(state["x"], state["cands"])
        cap = state["cands"].shape[0]
        return _on_host(state["cands"][:min(n, cap)], cap, n)
    if kind == "search":
        sp.single_pulse_search(state["x"], state["w"], 6.0, 8192, state["work"], state["cands"], state["count"])
        return _on_gpu(state["cands"], state["count"])
    if kind == "peaks":
        sp.single_pulse_search_window(state["x"], state["w"], 6.0, 8192, state["radius"], state["work"],
                                      state["cands"], state["count"])
        return _on_gpu(state["cands"], state["count"])
    if kind == "map":
        sp.best_snr_map(state["x"], state["w"], 8192, state["work"], state["best"], state["wbest"])
        return {"best": state["best"], "width": state["wbest"]}
    if kind == "batch":
        b = state["b"]
        b.run()
        return [_records(b.results(i), b.cap) for i in range(b.nbeams)]
    if kind == "stream":
        for b, g in enumerate(state["gulps"]):
            state["st"].push(b, g)
        done = sorted(state["st"].drain(), key=lambda r: r[0].beam)
        return [_records(c, state["st"].cap) for r, c in done]
    if kind in ("classify", "peaks_cls"):
        sub = state["sub"] if kind == "classify" else sp.cnn_extract(
            state["plan"], state["staged"], state["n_in"], state["cands"], POW2, t_in=state["t_in"])
        sp.cnn_features(sub, state["shift"], state["ft"], state["dmt"], state["work"])
        state["clf"].forward(state["ft"], state["dmt"], state["prob"])
        out = {"ft": state["ft"], "dmt": state["dmt"], "prob": state["prob"]}
        return out if kind == "classify" else dict(out, sub=sub)
    loss = state["clf"].backward(state["ft"], state["dmt"], state["labels"])
    return {"loss": loss, "grads": state["clf"].grads()}


# ------------------------------------------------------------------- work --
def work(case):
    """Bytes: inputs once, outputs once.  Flops: for the integer transforms
    the adds that even a perfect sharing of partial sums needs (one per input
    sample and per output sum); for the network its multiply-adds."""
    kind = case["kind"]
    net = sum(2 * 9 * ci * co * (128 >> l) ** 2 for l, (ci, co) in enumerate(zip(CIN, COUT))) * 2
    if kind in ("dmt", "beam", "beam_host", "stream", "batch", "peaks_cls"):
        if kind == "batch":
            beams = [(n, "steps", m) for n, m in zip(_ints(case["n_outs"]), _ints(case["max_dms"]))]
        else:
            beams = [(case["n_out"], case["dms"], case["max_dm"])] * case.get("beams", 1)
        if kind == "peaks_cls":
            per = 256 * case["t_in"]
            read = case["ncand"] * per * (case["nchan"] // 256)
            return {"bytes": read + case["ncand"] * (4 * per + 4 * 65536), "flops": case["ncand"] * (net + 2 * 65536 * 256)}
        nbytes = flops = 0
        for n, dms, m in beams:
            n_in, ndm = n + max_delay(case["nchan"], dms, m), trial_dms(dms, m).size
            nbytes += n_in * case["nchan"] + (ndm * n * 4 if kind == "dmt" else 0)
            flops += n_in * case["nchan"] + ndm * n * (1 + case.get("nw", 0))
        return {"bytes": nbytes, "flops": flops}
    if kind in ("search", "peaks", "map"):
        n = case["ndm"] * case["n_out"]
        return {"bytes": n * (9 if kind == "map" else 4), "flops": n * 3 * case["nw"]}
    if kind == "classify":
        b = case["batch"]
        return {"bytes": b * (256 * case["t_in"] * 4 + 2 * 65536 * 2 + 4), "flops": b * (net + 65536 * 256)}
    return {"bytes": case["batch"] * 2 * 65536 * 2 + 2 * 4 * make_params(0).size, "flops": 3 * case["batch"] * net}


# ------------------------------------------------------------------ exact --
def _exact_dmt(case, seed):
    n_out = case["n_out"]
    dms, f = trial_dms(case["dms"], case["max_dm"]), freqs(case["nchan"])
    n_in = n_out + max_delay(case["nchan"], case["dms"], case["max_dm"])
    if case["nchan"] * dms.size * n_out > 3e10:
        return None
    x = make_beam(seed, case["nchan"], n_in, n_out, case["max_dm"]).t().contiguous().to(torch.int32)
    t = torch.arange(n_out, device="cuda")
    out = torch.empty((dms.size, n_out), dtype=torch.int64, device="cuda")
    for d, dm in enumerate(dms):
        delay = np.floor(KDM * dm * (1.0 / (f * f) - 1.0 / (f[0] * f[0])) / TSAMP + 0.5).astype(np.int64)
        at = torch.as_tensor(delay, device="cuda")[:, None] + t[None, :]
        out[d] = x.gather(1, at).sum(dim=0)
    return out.to(torch.int32)


def _exact_map(case, seed):
    x = make_dmt(seed, case["ndm"], case["n_out"], case["nchan"]).double()
    n_out, L = case["n_out"], 8192
    nblk = max(1, n_out // L)
    block = torch.clamp(torch.arange(n_out, device="cuda") // L, max=nblk - 1)
    mean, std = torch.empty_like(x), torch.empty_like(x)
    for b in range(nblk):
        m = block == b
        mean[:, m] = x[:, m].mean(dim=1, keepdim=True)
        std[:, m] = x[:, m].std(dim=1, keepdim=True, unbiased=False)
    cs = torch.cat([torch.zeros_like(x[:, :1]), x.cumsum(dim=1)], dim=1)
    best = torch.full_like(x, -math.inf)
    for w in _widths(case):
        n = n_out - int(w) + 1
        s = cs[:, int(w):] - cs[:, :n]
        snr = (s - int(w) * mean[:, :n]) / (math.sqrt(int(w)) * std[:, :n])
        best[:, :n] = torch.maximum(best[:, :n], snr)
    return {"best": best, "width": None}


def _net(flat, img):
    k, x = 0, img[:, None]
    for ci, co in zip(CIN, COUT):
        w = flat[k:k + co * 9 * ci].view(co, 3, 3, ci).permute(0, 3, 1, 2)
        k += co * 9 * ci
        x = torch.relu(torch.nn.functional.conv2d(x, w, flat[k:k + co], stride=2, padding=1))
        k += co
    return x.mean(dim=(2, 3)) @ flat[k:k + FEAT] + flat[k + FEAT]


def _branches(seed):
    flat = torch.as_tensor(make_params(seed), device="cuda").double()
    return flat, flat.numel() // 2


def _exact_classify(case, seed):
    t_in = case["t_in"]
    sub = make_spectra(seed, case["batch"], t_in).double()
    f = freqs(4096).reshape(256, -1).mean(axis=1)
    k = f ** -2.0
    g = (k - k[0]) / (k[-1] - k[0])
    u0, B = (t_in - 256) // 2, case["batch"]
    ft = sub[:, :, u0:u0 + 256].clone()
    dmt = torch.zeros_like(ft)
    pad = torch.nn.functional.pad(sub, (256, 256))
    u = torch.arange(256, device="cuda")
    for j in range(256):
        sweep = ((t_in - 256) // 2) * (2.0 * j / 255.0 - 1.0)
        s = torch.as_tensor((np.sign(sweep * g) * np.floor(np.abs(sweep * g) + 0.5)).astype(np.int64), device="cuda")
        at = (256 + u0 + s)[:, None] + u[None, :]
        dmt[:, j] = pad.gather(2, at[None].expand(B, -1, -1)).sum(dim=1)
    out = []
    for x in (ft, dmt):
        x -= x.mean(dim=(1, 2), keepdim=True)
        x /= x.std(dim=(1, 2), keepdim=True, unbiased=False)
        out.append(x)
    flat, h = _branches(seed)
    p = torch.cat([torch.sigmoid(_net(flat[:h], a)) * torch.sigmoid(_net(flat[h:], b))
                   for a, b in zip(out[0].split(32), out[1].split(32))])
    return {"ft": out[0], "dmt": out[1], "prob": p}


def _exact_train(case, seed):
    ft, dmt, labels = make_images(seed, case["batch"])
    flat, h = _branches(seed)
    grad, loss = torch.zeros_like(flat), 0.0
    for a, b, y in zip(ft.double().split(16), dmt.double().split(16), labels.double().split(16)):
        w = flat.clone().requires_grad_(True)
        z1, z2 = _net(w[:h], a), _net(w[h:], b)
        lp = torch.nn.functional.logsigmoid(z1) + torch.nn.functional.logsigmoid(z2)
        part = -(y * lp + (1.0 - y) * torch.log(-torch.expm1(lp))).sum() / case["batch"]
        part.backward()
        grad += w.grad
        loss += float(part)
    return {"loss": loss, "grads": grad.cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "dmt":
        return _exact_dmt(case, seed)
    if kind == "map":
        return _exact_map(case, seed)
    if kind == "classify":
        return _exact_classify(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return None
