"""The measured cases: what a user of the library runs, through its public entry points.

Every family is one kind of work of the paper's setup (Sec. 2.2, Sec. 3): jobs of electrons in a prescribed
pulse (1D, reflected, 2D focus), many runs in one batch, a job driven one step per call, the 1D PIC, the
mono-energetic bunch in solid matter, the conversion of emitted photons to pairs, and the spectra and maps that
end a job.  Sizes are those of paper_1612_07592_gb300/workloads.py and of the tests, shortened where a whole job
would take long.  A pass of a job draws its initial state, steps, and forms the diagnostics, as a user's job does.

Photon and pair records leave the kernels in no particular order, so a pass returns them in a defined one: photons
sorted by (step, id), pairs at the place of their photon; the larger jobs return the photon map instead.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1612_07592_gb300 as pe
from paper_1612_07592_gb300 import workloads as W

AL, AU = W.AL, W.AU
CUDA = "cuda"
MAP_X, MAP_E, SPEC = 128, 64, 200            # bins of the photon map and of the electron spectrum


# ------------------------------------------------------------------------------------------------ the cases
def listed():
    return [
        # the paper's smallest job as the reference arithmetic: FP64, 1D Al, a0 = 27 (1e21 W/cm^2)
        dict(name="f64-1d-al-a27", family="job", precision="f64", field="plane", cp=False, a0=27.0, target="al",
             init="rest", n=10_000, steps=2000, x0_um=2.0, brems="direct", box=False),
        # the same job in FP32: a small request, one warp or less per scheduler, so the latency of a step counts
        dict(name="f32-1d-al-a27-small", family="job", precision="f32", field="plane", cp=False, a0=27.0, target="al",
             init="rest", n=10_007, steps=2000, x0_um=2.0, brems="direct", box=False),
        # the headline job: 1D Au, a0 = 270, Maxwell-Juttner start, 1e6 electrons x 4000 steps
        dict(name="f32-1d-au-a270", family="job", precision="f32", field="plane", cp=False, a0=270.0, target="au",
             init="mj", n=1_000_000, steps=4000, x0_um=2.0, brems="direct", box=False),
        # the 2D focus, circular polarisation, a0 = 855 per component
        dict(name="f32-2d-cp-a855", family="job", precision="f32", field="gauss", cp=True, a0=855.0, target="au",
             init="rest", n=2_000_003, steps=1000, x0_um=2.0, brems="direct", box=False),
        # a reflecting target: the electrons radiate in the standing wave, an emission in some per cent of the steps
        dict(name="f32-reflected-a270", family="job", precision="f32", field="reflected", cp=False, a0=270.0,
             target="au", init="mj", n=250_000, steps=3000, x0_um=2.0, brems="direct", box=False),
        # a host code that resumes a checkpoint and advances it one step per call
        dict(name="f32-one-step-calls", family="stepwise", cp=False, a0=270.0, target="au", n=6_000_001, before=260,
             steps=20),
        # a parameter scan in one batch: 64 targets and intensities, uneven sizes
        dict(name="f32-batch-64", family="batch", runs=64, median=50_000, steps=1000),
        # the self-consistent 1D PIC around the step
        dict(name="f32-pic-1d-au", family="pic", precision="f32", cp=False, a0=270.0, n=1_000_000, n_cells=1000,
             steps=500, x0_um=2.0),
        # the paper's own benchmark of the bremsstrahlung module: 1 GeV electrons through Au, fields off
        dict(name="f32-bunch-1gev-au", family="bunch", E0_mev=1000.0, target="Au", n=500_009, steps=2000, dt=1.0,
             brems="direct"),
        # Bethe-Heitler conversion of photons on their way through the rest of the target
        dict(name="bh-pairs-au", family="bh", target="Au", n=300_001, steps=2000, method="direct"),
        # Breit-Wheeler conversion of energetic photons that meet the pulse and its reflection
        dict(name="f32-bw-pairs-reflected", family="bw", precision="f32", field="reflected", cp=False, a0=400.0,
             n=400_003, steps=2000),
        # what ends a job: the electron spectrum and the photon map of its state
        dict(name="spectra-of-a-job", family="diag", n=3_000_000, steps=700, nx=200, ne=64, n_bins=200),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["job", "job", "job", "job", "stepwise", "batch", "pic", "bunch", "bh", "bw", "diag"])
    target = rng.choice(["al", "au"])
    if family == "job":
        precision = rng.choice(["f32", "f32", "f32", "f64"])
        field = rng.choice(["plane", "plane", "reflected", "gauss"])
        steps = _log_int(rng, 300, 4000)
        # particle-steps: up to those of the headline job (1D), of the shorter 2D and reflected ones, and of 2e8 in FP64
        most = 2e8 if precision == "f64" else {"plane": 4e9, "reflected": 7e8, "gauss": 2e9}[field]
        n = min(_log_int(rng, 1_000, 2_000_000), int(most / steps))
        return dict(family="job", precision=precision, field=field, cp=rng.random() < 0.4,
                    a0=math.exp(rng.uniform(math.log(27.0), math.log(855.0))), target=target,
                    init=rng.choice(["rest", "mj"]), n=n, steps=steps, x0_um=rng.choice([0.5, 1.0, 2.0]),
                    brems=rng.choice(["direct", "direct", "null"]), box=rng.random() < 0.2)
    if family == "stepwise":
        return dict(family=family, cp=rng.random() < 0.4, a0=rng.uniform(27.0, 400.0), target=target,
                    n=_log_int(rng, 1_000, 6_000_000), before=rng.randint(200, 400), steps=rng.randint(1, 20))
    if family == "batch":
        return dict(family=family, runs=rng.randint(2, 64), median=_log_int(rng, 2_000, 50_000),
                    steps=rng.randint(300, 1000))
    if family == "pic":
        return dict(family=family, precision=rng.choice(["f32", "f32", "f64"]), cp=rng.random() < 0.4,
                    a0=rng.uniform(27.0, 400.0), n=_log_int(rng, 5_000, 200_000), n_cells=rng.randint(400, 2000),
                    steps=rng.randint(250, 500), x0_um=rng.choice([1.0, 2.0]))
    if family == "bunch":
        return dict(family=family, E0_mev=rng.choice([100.0, 500.0, 1000.0]), target=rng.choice(["Al", "Au"]),
                    n=_log_int(rng, 10_000, 500_000), steps=rng.randint(300, 2000), dt=rng.choice([0.1, 1.0]),
                    brems=rng.choice(["direct", "null"]))
    if family == "bh":
        return dict(family=family, target=rng.choice(["Al", "Au"]), n=_log_int(rng, 3_000, 300_000),
                    steps=rng.randint(300, 2000), method=rng.choice(["direct", "free"]))
    if family == "bw":
        return dict(family=family, precision=rng.choice(["f32", "f32", "f64"]),
                    field=rng.choice(["plane", "reflected", "gauss"]), cp=rng.random() < 0.4,
                    a0=rng.uniform(100.0, 400.0), n=_log_int(rng, 3_000, 60_000), steps=rng.randint(300, 2000))
    return dict(family=family, n=_log_int(rng, 30_000, 3_000_000), steps=rng.randint(300, 700),
                nx=rng.randint(50, 400), ne=rng.randint(32, 128), n_bins=rng.randint(50, 1000))


# ------------------------------------------------------------------------------------------------ preparing
_tables: dict = {}


def _table_set(large=True):
    """The sampling tables of the library, built once per program as a user's program does."""
    if large not in _tables:
        d = W.tables_large() if large else W.tables_small()
        _tables[large] = pe.pe_create_tables(d, (13.0, 79.0))
    return _tables[large]


def _bw_set():
    if "bw" not in _tables:
        _tables["bw"] = pe.pe_bw_tables_create()
    return _tables["bw"]


def _run_dict(case, seed):
    """The run of a case as workloads.base_run describes it."""
    f = case["family"]
    if f == "bunch":
        d = dict(W.bunch(case["E0_mev"], case["target"], thickness_m=5e-3, dt_over_T=case["dt"])["run"])
        d.update(seed=seed, brems_method=int(case["brems"] == "null"))
        return d
    if f == "bh":
        d = dict(W.bunch(1000.0, case["target"], thickness_m=1.5e-3)["run"])
        d.update(seed=seed)
        return d
    if f == "diag":
        return W.base_run(a0=270.0, init_dist=1, T_mev=1.0, seed=seed, slab_x0_m=0.5e-6, **AU)
    if f == "bw":
        d = W.base_run(a0=case["a0"], polarisation=int(case["cp"]), geometry=int(case["field"] == "gauss"), seed=seed,
                       **AU)
        if case["field"] == "reflected":
            d.update(reflect_r=1.0, mirror_x_m=3e-6)
        return d
    target = AL if case.get("target") == "al" else AU
    if f == "stepwise":
        return W.base_run(a0=case["a0"], polarisation=int(case["cp"]), init_dist=1, T_mev=1.0, seed=seed, **target)
    x0 = case["x0_um"] * 1e-6
    d = W.base_run(a0=case["a0"], polarisation=int(case["cp"]), seed=seed, slab_x0_m=x0, focus_x_m=x0, **target)
    if f == "pic":
        d.update(init_dist=1, T_mev=1.0, geometry=pe.PE_PIC_1D, n_cells=case["n_cells"])
        return d
    d.update(init_dist=int(case["init"] == "mj"), geometry=int(case["field"] == "gauss"),
             brems_method=int(case["brems"] == "null"))
    if case["field"] == "gauss":
        d.update(slab_thick_m=2e-6, y_half_m=3e-6)
    if case["field"] == "reflected":
        d.update(reflect_r=1.0, mirror_x_m=x0 + 1e-6)
    if case["box"]:
        d.update(box_enable=1, box_x_m=(0.0, x0 + 4e-6))
    return d


def _precision(case):
    return pe.PE_F64 if case.get("precision") == "f64" else pe.PE_F32


class Job:
    """Parameters and buffers of one run: what a program holds before it starts the run."""

    def __init__(self, run, precision, n, capacity, events=False):
        self.params = pe.run_params(precision=precision, **run)
        self.f32 = precision == pe.PE_F32
        self.n, self.capacity = n, capacity
        dt = torch.float32 if self.f32 else torch.float64
        self.x, self.y, self.tau = (torch.zeros(n, dtype=torch.float64, device=CUDA) for _ in range(3))
        self.u = [torch.zeros(n, dtype=dt, device=CUDA) for _ in range(3)]
        self.photons = torch.zeros(max(capacity, 1), 8, dtype=torch.int32, device=CUDA)
        self.hist = torch.zeros(pe.HIST_WORDS, dtype=torch.int64, device=CUDA)
        self.tally = torch.zeros(pe.TALLY_WORDS, dtype=torch.int64, device=CUDA)
        self.events = torch.zeros(n, dtype=torch.int64, device=CUDA) if events else None
        self.wait = (torch.zeros(n, dtype=torch.int32, device=CUDA)
                     if self.params.brems_method == pe.PE_BREMS_NULL else None)
        self.grid = (torch.zeros(pe.pic_grid_words(self.params.n_cells), dtype=dt, device=CUDA)
                     if self.params.geometry == pe.PE_PIC_1D else None)
        self.spectrum = torch.zeros(SPEC, dtype=torch.int64, device=CUDA)
        self.map = torch.zeros(MAP_X * MAP_E, dtype=torch.int64, device=CUDA)

    def buffers(self):
        def p(t):
            return None if t is None else t.data_ptr()
        return pe.Buffers(p(self.x), p(self.y), p(self.u[0]), p(self.u[1]), p(self.u[2]), p(self.tau), p(self.photons),
                          self.capacity, p(self.hist), p(self.tally), p(self.events), p(self.wait), p(self.grid))

    def state(self):
        """The state by name; FP32 positions and optical depths as their (hi, lo) parts."""
        out = {}
        for name, t in (("x", self.x), ("y", self.y), ("tau", self.tau)):
            if name == "y" and self.params.geometry != pe.PE_GAUSS_2D:
                continue
            if self.f32:
                pair = t.view(torch.float32).view(-1, 2)
                out[name], out[name + "_lo"] = pair[:, 0], pair[:, 1]
            else:
                out[name] = t
        out.update(ux=self.u[0], uy=self.u[1], uz=self.u[2])
        return out

    def results(self):
        out = dict(state=self.state(), hist=self.hist, tally=self.tally)
        for name in ("events", "wait", "grid"):
            if getattr(self, name) is not None:
                out[name] = getattr(self, name)
        return out

    def sorted_photons(self):
        """The stored photons in order of (step, id); rows past the count are zero."""
        p = self.photons
        got = torch.arange(self.capacity, device=CUDA) < self.tally[pe.T["N_PHOTONS"]]
        key = (p[:, 6].long() << 32) | (p[:, 7].long() & 0xFFFFFFFF)
        order = torch.where(got, key, torch.iinfo(torch.int64).max).argsort()
        p = torch.where(got[:, None], p, 0)[order]
        return dict(values=p[:, :6].contiguous().view(torch.float32), words=p[:, 6:])

    def diagnostics(self, handle):
        x0, L = self.params.slab_x0_m, 12e-6
        pe.pe_electron_spectrum(handle, SPEC, 0.01, 1e4, self.spectrum.data_ptr())
        pe.pe_photon_map(handle, MAP_X, x0 - 1e-6, x0 + L, MAP_E, 0.511, 1e4, self.map.data_ptr())
        return dict(spectrum=self.spectrum, photon_map=self.map)


def _stream():
    return torch.cuda.current_stream().cuda_stream


def _photon_room(case):
    """Photon slots of a job, above what it can emit (a job at full length: up to some hundred per electron)."""
    n, steps = case["n"], case["steps"]
    if case["family"] in ("bunch", "pic"):
        return 24 * n
    per = {"reflected": 0.08 * steps, "plane": 0.01 * steps, "gauss": 0.02 * steps}[case.get("field", "plane")]
    return int(min(n * max(per, 4.0), 6e7 if n > 30_000 else 4e6))


def prepare(case, seed):
    f = case["family"]
    s = dict(case=case, family=f)
    if f in ("job", "pic", "bunch"):
        s["tables"] = _table_set(f != "bunch" and case.get("target") != "al")
        s["job"] = Job(_run_dict(case, seed), _precision(case), case["n"], _photon_room(case),
                       events=f == "job" and case["n"] <= 30_000)
    elif f == "stepwise":
        # a checkpoint: the state that the run reached at step `before`, and the buffers it is resumed in
        s["tables"] = _table_set()
        job = s["job"] = Job(_run_dict(case, seed), pe.PE_F32, case["n"], 4 * case["n"])
        h = pe.pe_init_particles(s["tables"], job.params, job.n, job.buffers(), _stream())
        pe.pe_step([h], case["before"])
        pe.pe_destroy(h)
        s["live"] = [job.x, job.tau, *job.u, job.hist, job.tally]
        s["saved"] = [t.clone() for t in s["live"]]
    elif f == "batch":
        s["tables"] = _table_set()
        s["jobs"], s["out"] = _batch(case, seed)
    elif f in ("bh", "bw"):
        s["tables"] = _table_set(False)
        s["bw"] = _bw_set() if f == "bw" else None
        # the run whose target, fields and steps the photons cross; its own electrons are not what is measured
        job = s["job"] = Job(_run_dict(case, seed), _precision(case), 256, 1 << 16)
        s["handle"] = pe.pe_init_particles(s["tables"], job.params, job.n, job.buffers(), _stream())
        pe.pe_step([s["handle"]], case["steps"])
        n, cap = case["n"], case["n"]
        s["photons"] = _photons(case, seed)
        s["pairs"] = torch.zeros(cap, 10, dtype=torch.int32, device=CUDA)
        s["place"] = torch.arange(cap, device=CUDA)
        s["counts"] = torch.zeros(pe.PAIR_TALLY_WORDS, dtype=torch.int64, device=CUDA)
    else:
        s["tables"] = _table_set()
        job = s["job"] = Job(_run_dict(case, seed), pe.PE_F32, case["n"], 4 * case["n"])
        s["handle"] = pe.pe_init_particles(s["tables"], job.params, job.n, job.buffers(), _stream())
        pe.pe_step([s["handle"]], case["steps"])
        s["spectrum"] = torch.zeros(case["n_bins"], dtype=torch.int64, device=CUDA)
        s["map"] = torch.zeros(case["nx"] * case["ne"], dtype=torch.int64, device=CUDA)
    torch.cuda.synchronize()
    return s


def _batch(case, seed):
    """Runs of one scan in shared arrays: run k takes the elements at[k] .. at[k] + n[k]."""
    k, rng = case["runs"], np.random.default_rng(case["runs"])        # the sizes are the scan's, not the seed's
    n = np.clip(np.round(np.exp(np.log(case["median"]) + rng.standard_normal(k))), 500, 8 * case["median"]).astype(int)
    n = (n * min(1.0, 1.6 * case["median"] * k / n.sum())).astype(int) | 1
    at = np.concatenate([[0], np.cumsum((n + 3) & ~3)])
    m = int(at[-1])
    x, y, tau = (torch.zeros(m, dtype=torch.float64, device=CUDA) for _ in range(3))
    u = [torch.zeros(m, dtype=torch.float32, device=CUDA) for _ in range(3)]
    photons = torch.zeros(40 * m, 8, dtype=torch.int32, device=CUDA)
    hist = torch.zeros(k, pe.HIST_WORDS, dtype=torch.int64, device=CUDA)
    tally = torch.zeros(k, pe.TALLY_WORDS, dtype=torch.int64, device=CUDA)
    jobs = []
    for i in range(k):
        run = W.base_run(a0=W.a0_of(10.0 ** (21 + 3 * i / max(k - 1, 1))), run_id=i, seed=seed,
                         **(AL if i % 2 == 0 else AU))
        a = int(at[i])
        b = pe.Buffers(x[a:].data_ptr(), y[a:].data_ptr(), *(v[a:].data_ptr() for v in u), tau[a:].data_ptr(),
                       photons[40 * a:].data_ptr(), 40 * int(n[i]), hist[i].data_ptr(), tally[i].data_ptr(), None, None,
                       None)
        jobs.append((pe.run_params(precision=pe.PE_F32, **run), int(n[i]), b))
    keep = torch.zeros(m, dtype=torch.bool, device=CUDA)
    for i in range(k):
        keep[int(at[i]):int(at[i]) + int(n[i])] = True
    xs, ts = x.view(torch.float32).view(-1, 2), tau.view(torch.float32).view(-1, 2)
    out = dict(x=xs[:, 0], x_lo=xs[:, 1], tau=ts[:, 0], tau_lo=ts[:, 1], ux=u[0], uy=u[1], uz=u[2], hist=hist,
               tally=tally)
    return jobs, dict(out, photons=photons, keep=keep)


def _photons(case, seed):
    kl = 2.0 * math.pi / W.LAMBDA
    if case["family"] == "bh":
        # the bremsstrahlung photons of the bunch: forward, emitted along the first half of the crossing
        p = W.synthetic_photons(case["n"], seed, (0.0, 0.4 * case["steps"] * 2 * math.pi), (2.0, 2000.0),
                                (0, case["steps"] // 2), theta_max=0.05, mech_frac=1.0)
    else:
        p = W.synthetic_photons(case["n"], seed, (1e-6 * kl, 4e-6 * kl), (100.0, 20000.0), (0, case["steps"] // 2),
                                theta_max=0.6, y_half=2e-6 * kl if case["field"] == "gauss" else 0.0)
    return torch.from_numpy(p.view(np.int32).reshape(-1, 8)).to(CUDA)


# ------------------------------------------------------------------------------------------------ one pass
def run(s):
    f = s["family"]
    case = s["case"]
    if f in ("job", "pic", "bunch"):
        job = s["job"]
        h = pe.pe_init_particles(s["tables"], job.params, job.n, job.buffers(), _stream())
        pe.pe_step([h], case["steps"])
        out = job.results()
        if job.events is not None:
            out["photons"] = job.sorted_photons()
        else:
            out.update(job.diagnostics(h))
        pe.pe_destroy(h)
        return out
    if f == "stepwise":
        job = s["job"]
        for t, v in zip(s["live"], s["saved"]):
            t.copy_(v)
        h = pe.pe_resume_particles(s["tables"], job.params, job.n, job.buffers(), case["before"], _stream())
        for _ in range(case["steps"]):
            pe.pe_step([h], 1)
        pe.pe_destroy(h)
        return job.results()
    if f == "batch":
        hs = [pe.pe_init_particles(s["tables"], p, n, b, _stream()) for p, n, b in s["jobs"]]
        pe.pe_step(hs, case["steps"])
        for h in hs:
            pe.pe_destroy(h)
        return {k: v for k, v in s["out"].items() if k not in ("photons", "keep")}
    if f in ("bh", "bw"):
        n, pairs, counts = case["n"], s["pairs"], s["counts"]
        if f == "bh":
            method = pe.PE_PAIR_DIRECT if case["method"] == "direct" else pe.PE_PAIR_FREE_PATH
            pe.pe_pair_transport(s["handle"], s["photons"].data_ptr(), n, -1, pairs.data_ptr(), len(pairs),
                                 counts.data_ptr(), method)
        else:
            pe.pe_bw_transport(s["handle"], s["bw"], s["photons"].data_ptr(), n, -1, pairs.data_ptr(), len(pairs),
                               counts.data_ptr())
        # each pair at its photon's place
        at = torch.where(s["place"] < counts[0], pairs[:, 8].long(), n)
        by_photon = torch.zeros(n + 1, 10, dtype=torch.int32, device=CUDA)
        by_photon[at] = pairs
        by_photon = by_photon[:n]
        return dict(values=by_photon[:, :7].contiguous().view(torch.float32), words=by_photon[:, 7:], counts=counts)
    pe.pe_electron_spectrum(s["handle"], case["n_bins"], 0.01, 1e4, s["spectrum"].data_ptr())
    pe.pe_photon_map(s["handle"], case["nx"], -0.5e-6, 8e-6, case["ne"], 0.511, 1e4, s["map"].data_ptr())
    return dict(spectrum=s["spectrum"], photon_map=s["map"])


# ------------------------------------------------------------------------------------------------ its work
# Single operations of one electron in one step: field, push, eta, rate, position (two pulses for the reflected
# wave; envelope, curvature and Gouy phase in 2D; none but the push with constant fields), the test of Eq. 4 in the target.
_STEP = {"plane": 124, "reflected": 200, "gauss": 250, "const": 70, "pic": 140}


def work(case):
    f = case["family"]
    if f in ("job", "pic", "bunch", "stepwise", "diag"):
        n, word = case["n"], 8 if case.get("precision") == "f64" else 4
        state = n * (2 * 8 + 3 * word + (8 if case.get("field") == "gauss" else 0))
        if f == "diag":
            return dict(bytes=n * (8 + 3 * 4) + 8 * (case["nx"] * case["ne"] + case["n_bins"]), flops=40 * n)
        kind = {"job": case.get("field"), "pic": "pic", "bunch": "const", "stepwise": "plane"}[f]
        # a job writes its state once; single-step calls read and write it in every one, the PIC holds it in between
        bytes_ = state * (2 * case["steps"] if f == "stepwise" else 1)
        return dict(bytes=bytes_, flops=_STEP[kind] * n * case["steps"])
    if f == "batch":
        n = 1.5 * case["median"] * case["runs"]
        return dict(bytes=28 * n, flops=_STEP["plane"] * n * case["steps"])
    per = 60 if f == "bh" else 150
    return dict(bytes=case["n"] * 32.0, flops=per * case["n"] * case["steps"] * 0.4)


# ------------------------------------------------------------------------------------------------ in 64 bits
# The step, its tables and its draws in plain float64 torch, for the runs in which a rounding does not grow into
# another history: emissions are drawn events, and in the longer runs at a0 = 270 and above (1D, reflected, PIC) a
# last-bit change of one momentum moves later emissions, so their states have no counterpart in other arithmetic.
ALPHA, RE, ME, HBC, C0 = 7.2973525693e-3, 2.8179403262e-15, 0.51099895, 197.3269804e-15, 299792458.0


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.tensor(0.5 * (x + 1.0), device=CUDA), torch.tensor(0.5 * w, device=CUDA)


def _bessel(nu, y, over=False):
    """K_nu(y), or with `over` its integral from y to infinity, by the trapezoid rule on int exp(-y cosh t) cosh(nu t)."""
    top = torch.acosh(1.0 + 760.0 / y) + 1.0
    m = 1200
    t = torch.linspace(0.0, 1.0, m, dtype=torch.float64, device=CUDA) * top[:, None]
    g = torch.exp(-y[:, None] * torch.cosh(t) + nu * t) * 0.5 * (1.0 + torch.exp(-2.0 * nu * t))
    if over:
        g = g / torch.cosh(t)
    g[:, 0] *= 0.5
    return g.sum(1) * top / (m - 1)


def _log_grid(lo, hi, n):
    return torch.exp(torch.linspace(math.log(lo), math.log(hi), n, dtype=torch.float64, device=CUDA))


_model: dict = {}


def _ncs_tables(p):
    gx, gw = _gauss(8)
    ly, lq = math.log(p["y_min"]), math.log(p["y_min"] * 1e-8)
    edges = torch.cat([torch.linspace(lq, ly, 41, dtype=torch.float64, device=CUDA)[:-1],
                       torch.linspace(ly, math.log(p["y_max"]), p["n_y"], dtype=torch.float64, device=CUDA)])
    d = edges[1:] - edges[:-1]
    y = torch.exp(edges[:-1, None] + gx * d[:, None])
    k23, ik53 = (_bessel(nu, y.reshape(-1), o).view_as(y) for nu, o in ((2 / 3, False), (5 / 3, True)))
    eta = _log_grid(p["eta_min"], p["eta_max"], p["n_eta"])

    def cells(e):
        q = 3.0 * e * y
        dl = q / (2.0 + q)
        return ((dl * dl * y * k23 + (1.0 - dl) * y * ik53) * 2.0 / (2.0 + q) * gw * d[:, None]).sum(1)

    rows = torch.stack([cells(e) for e in eta] + [cells(0.0 * eta[0])])
    y0 = torch.exp(edges[:1])
    rows[:, 0] += 3.0 * (y0 * _bessel(5 / 3, y0, True))
    cum = rows.cumsum(1)[:, 39:]
    return cum[:-1, -1].clone(), cum / cum[:, -1:]


def _screen(Z, g, e):
    a2 = (ALPHA * Z) ** 2
    f = a2 * (1 / (1 + a2) + 0.20206 - 0.0369 * a2 + 0.0083 * a2 ** 2 - 0.002 * a2 ** 3)
    phi1 = 20.863 - 2 * torch.log1p((0.55846 * g) ** 2) - 4 * (1 - 0.6 * torch.exp(-0.9 * g) - 0.4 * torch.exp(-1.5 * g))
    psi1 = 28.340 - 2 * torch.log1p((3.621 * e) ** 2) - 4 * (1 - 0.7 * torch.exp(-8 * e) - 0.3 * torch.exp(-29.2 * e))
    dphi, dpsi, lz = (2 / 3) / (1 + 6.5 * g + 6 * g * g), (2 / 3) / (1 + 40 * e + 400 * e * e), math.log(Z)
    return (Z * Z * (phi1 - 4 / 3 * lz - 4 * f) + Z * (psi1 - 8 / 3 * lz)), Z * Z * dphi + Z * dpsi


def _cumulated(cells):
    cum = torch.cat([torch.zeros_like(cells[:, :1]), cells.cumsum(1)], 1)
    flat = torch.linspace(0, 1, cum.shape[1], dtype=torch.float64, device=CUDA)
    return cum[:, -1].clone(), torch.where(cum[:, -1:] > 0, cum / cum[:, -1:], flat)


def _brems_tables(p, Z):
    gx, gw = _gauss(16)
    n = p["n_s"]
    g = _log_grid(p["gamma_min"], p["gamma_max"], p["n_E"])[:, None, None]
    s = (torch.arange(n - 1, device=CUDA)[:, None] + gx) / (n - 1)
    ycut, ymax = p["photon_min_mc2"] / g, 1.0 - 1.0 / g
    L = torch.log(ymax / ycut).clamp(min=0.0)
    y = ycut * torch.exp(s * L)
    v = 100 * y / (g * (1 - y))
    main, diff = _screen(Z, v / Z ** (1 / 3), v / Z ** (2 / 3))
    dcs = (4 / 3 - 4 / 3 * y + y * y) * main + (2 / 3) * (1 - y) * diff
    return _cumulated((dcs.clamp(min=0.0) * L * gw / (n - 1)).sum(2))


def _bh_tables(p, Z):
    gx, gw = _gauss(16)
    n = p["n_s"]
    k = _log_grid(2.0, p["gamma_max"], p["n_E"])[:, None, None]
    s = (torch.arange(n - 1, device=CUDA)[:, None] + gx) / (n - 1)
    span = 1.0 - 2.0 / k
    x = 1.0 / k + s * span
    xx = x * (1.0 - x)
    v = 100.0 / (k * xx)
    main, diff = _screen(Z, v / Z ** (1 / 3), v / Z ** (2 / 3))
    dcs = (1 - 4 / 3 * xx) * main - (2 / 3) * xx * diff
    return _cumulated((dcs.clamp(min=0.0) * span * gw / (n - 1)).sum(2))


def _tabs(large):
    if large not in _model:
        p = W.tables_large() if large else W.tables_small()
        h, cdf = _ncs_tables(p)
        _model[large] = dict(p=p, h=h, cdf=cdf, br={z: _brems_tables(p, z) for z in (13.0, 79.0)},
                             bh={z: _bh_tables(p, z) for z in (13.0, 79.0)})
    return _model[large]


def _row(v, lo, hi, n):
    t = ((torch.log(v) - math.log(lo)) * ((n - 1) / (math.log(hi) - math.log(lo)))).nan_to_num(0.0).clamp(0.0, n - 1.0)
    i = t.floor().clamp(max=n - 2).long()
    return i, t - i


def _invert(cdf, ia, ib, w, R):
    """Column and fraction of R in the interpolated rows; column -1 below the first node (fraction R / c_0)."""
    n = cdf.shape[1]
    lo, hi = torch.zeros_like(ia), torch.full_like(ia, n - 1)
    at = lambda j: (1 - w) * cdf[ia, j] + w * cdf[ib, j]  # noqa: E731
    c0 = at(lo)
    for _ in range(n.bit_length()):
        mid = (lo + hi) // 2
        up = (at(mid) <= R) & (hi - lo > 1)
        lo, hi = torch.where(up, mid, lo), torch.where(up | (hi - lo <= 1), hi, mid)
    cl, ch = at(lo), at(lo + 1)
    f = torch.where(ch > cl, (R - cl) / (ch - cl), 0.0).clamp(max=1.0)
    return torch.where(R < c0, -1, lo), torch.where(R < c0, R / c0, f)


def _philox(c0, c1, c2, c3, seed):
    M = 0xFFFFFFFF
    k0, k1 = seed & M, (seed >> 32) & M
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & M) ^ c1 ^ k0, b & M, ((a >> 32) & M) ^ c3 ^ k1, a & M
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    return c0, c1, c2, c3


def _uni53(lo, hi):
    return (((hi << 21) | (lo >> 11)).double() + 0.5) * 2.0 ** -53


def _uni32(v):
    return (v.double() + 0.5) * 2.0 ** -32


class Model:
    """A run in float64: initial draw and steps of the prescribed-field kinds, direct bremsstrahlung."""

    def __init__(self, d, n, tabs):
        self.d, self.n, self.t = d, n, tabs
        kl = 2 * math.pi / d["lambda_m"]
        self.kl, self.seed, self.dt = kl, d["seed"], d["dt_over_T"] * 2 * math.pi
        self.x0, self.x1, self.yh = d["slab_x0_m"] * kl, (d["slab_x0_m"] + d["slab_thick_m"]) * kl, d["y_half_m"] * kl
        self.ES = ME * d["lambda_m"] / (2 * math.pi * HBC)
        self.ncs = math.sqrt(3) * ALPHA / (2 * math.pi) * self.ES * self.dt
        self.K = (d["ne_over_nc"] * math.pi / (RE * d["lambda_m"] ** 2) / d["charge_state"] * ALPHA * RE ** 2
                  * self.dt / kl)
        self.pr = 2 * math.pi * d["ramp_periods"]
        self.pf = 2 * math.pi * d["flat_s"] * C0 / d["lambda_m"]
        self.id = torch.arange(n, device=CUDA)
        self.run_id = d.get("run_id", 0)
        self._init()

    def words(self, idx, step, purpose):
        i = self.id if idx is None else self.id[idx]
        z = torch.zeros_like(i)
        return _philox(i, z + self.run_id, z + step, z + purpose, self.seed)

    def _init(self):
        d, n = self.d, self.n
        w = self.words(None, 0, 2)
        self.tau = -torch.log(_uni53(w[0], w[1]))
        p = self.words(None, 0, 3)
        beam = d["init_dist"] == 2
        self.x = torch.full((n,), self.x0, dtype=torch.float64, device=CUDA) if beam else (
            self.x0 + (self.x1 - self.x0) * _uni32(p[0]))
        self.y = (-self.yh + 2 * self.yh * _uni32(p[1])) if d["geometry"] == 1 else torch.zeros_like(self.x)
        self.u = [torch.zeros_like(self.x) for _ in range(3)]
        if beam:
            self.u[0] += math.sqrt(d["beam_gamma"] ** 2 - 1)
        if d["init_dist"] == 1:
            th, um = d["T_mev"] / ME, torch.zeros_like(self.x)
            open_ = torch.ones_like(self.x, dtype=torch.bool)
            for r in range(64):
                X = [_uni32(v) for v in self.words(None, 0, 4 + r)]
                uu = -th * torch.log(X[0] * X[1] * X[2])
                ee = -th * torch.log(X[0] * X[1] * X[2] * X[3])
                ok = open_ & (ee * ee - uu * uu > 1)
                um, open_ = torch.where(ok, uu, um), open_ & ~ok
                if not open_.any():
                    break
            X5, ph = _uni32(p[2]), 2 * math.pi * _uni32(p[3])
            sn = 2 * torch.sqrt(X5 * (1 - X5))
            self.u = [um * (2 * X5 - 1), um * sn * torch.cos(ph), um * sn * torch.sin(ph)]

    def env(self, phi):
        rem = 2 * self.pr + self.pf - phi
        k = 0.5 * math.pi / self.pr
        a = (k * torch.minimum(phi, rem)).clamp(0.0, 0.5 * math.pi)
        s, c = torch.sin(a), torch.cos(a)
        return s * s, torch.copysign(2 * k * s * c, rem - phi)

    def plane(self, phi):
        g, dg = self.env(phi)
        s, c = torch.sin(phi), torch.cos(phi)
        ez = self.d["a0"] * (dg * c - g * s) if self.d["polarisation"] else torch.zeros_like(g)
        return -self.d["a0"] * (dg * s + g * c), ez

    def fields(self, x, y, t):
        d, z = self.d, torch.zeros_like(x)
        if d["geometry"] == 2:
            return [z, z, z], [z, z, z]
        if d["geometry"] == 0:
            ey, ez = self.plane(t - x)
            if not d.get("reflect_r", 0):
                return [z, ey, ez], [z, -ez, ey]
            ry, rz = (-d["reflect_r"] * v for v in self.plane(t + x - 2 * d["mirror_x_m"] * self.kl))
            return [z, ey + ry, ez + rz], [z, rz - ez, ey - ry]
        w0, xf, a0 = d["w0_m"] * self.kl, d["focus_x_m"] * self.kl, d["a0"]
        zr, xi = 0.5 * w0 * w0, x - xf
        w2 = w0 * w0 * (1 + (xi / zr) ** 2)
        iR, S = xi / (xi * xi + zr * zr), torch.sqrt(w0 / torch.sqrt(w2)) * torch.exp(-y * y / w2)
        phi = t - x
        g, dg = self.env(phi)
        th = phi - 0.5 * y * y * iR + 0.5 * torch.atan(xi / zr)
        s, c = torch.sin(th), torch.cos(th)
        ey, ex = -a0 * S * (dg * s + g * c), a0 * g * S * (y * iR * c + 2 * y / w2 * s)
        if not d["polarisation"]:
            return [ex, ey, z], [z, z, ey]
        ez = a0 * S * (dg * c - g * s)
        return [ex, ey, ez], [a0 * g * S * (2 * y / w2 * c - y * iR * s), -ez, ey]

    def chi(self, u, gamma, E, B, rest=1.0):
        """sqrt((gamma E + u x B)^2 - (u.E)^2) / E_S, arranged without the cancellation along +x."""
        gm = torch.where(u[0] > 0, (rest + u[1] ** 2 + u[2] ** 2) / (gamma + u[0]), gamma - u[0])
        d = [B[0], B[1] + E[2], B[2] - E[1]]
        V = [gm * E[0] + u[1] * d[2] - u[2] * d[1], gm * E[1] + u[2] * d[0] - u[0] * d[2],
             gm * E[2] + u[0] * d[1] - u[1] * d[0]]
        q = V[0] ** 2 + V[1] ** 2 + V[2] ** 2 + 2 * V[0] * (u[0] * E[0] + u[1] * E[1] + u[2] * E[2])
        return torch.sqrt(q.clamp(min=0)) / self.ES

    def recoil(self, i, gamma, w):
        um = torch.sqrt(sum(v[i] ** 2 for v in self.u))
        g2 = gamma[i] - w
        un = torch.sqrt((g2 * g2 - 1).clamp(min=0)) / um
        for v in self.u:
            v[i] *= un
        gamma[i] = torch.sqrt(1 + sum(v[i] ** 2 for v in self.u))

    def step(self, n):
        d, t, p, u, h = self.d, self.t, self.t["p"], self.u, 0.5 * self.dt
        E, B = self.fields(self.x, self.y, n * self.dt)
        if d["geometry"] != 2:
            um = [u[k] - h * E[k] for k in range(3)]
            ig = 1 / torch.sqrt(1 + sum(v * v for v in um))
            b = [-h * v * ig for v in B]
            f = 2 / (1 + sum(v * v for v in b))
            cross = lambda a, c: [a[1] * c[2] - a[2] * c[1], a[2] * c[0] - a[0] * c[2], a[0] * c[1] - a[1] * c[0]]  # noqa: E731
            q = [v + w for v, w in zip(um, cross(um, b))]
            self.u = u = [v + f * w - h * e for v, w, e in zip(um, cross(q, b), E)]
        gamma = torch.sqrt(1 + sum(v * v for v in u))
        if d["enable_ncs"]:
            eta = self.chi(u, gamma, E, B)
            i, w = _row(eta, p["eta_min"], p["eta_max"], p["n_eta"])
            hv = torch.where(eta >= p["eta_min"], (1 - w) * t["h"][i] + w * t["h"][i + 1], 5 * math.pi / 3)
            self.tau = self.tau - self.ncs * eta / gamma * hv
            k = (self.tau <= 0).nonzero()[:, 0]
            if len(k):
                a = self.words(k, n, 1)
                e, low = eta[k], eta[k] < p["eta_min"]
                j, fr = _invert(t["cdf"], torch.where(low, p["n_eta"], i[k]), torch.where(low, p["n_eta"], i[k] + 1),
                                w[k], _uni53(a[0], a[1]))
                dly = math.log(p["y_max"] / p["y_min"]) / (p["n_y"] - 1)
                y = torch.where(j < 0, p["y_min"] * fr ** 3, torch.exp(math.log(p["y_min"]) + (j + fr) * dly))
                q = 3 * e * y
                self.recoil(k, gamma, torch.minimum(q / (2 + q) * gamma[k], gamma[k] - 1))
                self.tau[k] = -torch.log(_uni53(a[2], a[3]))
        if d["enable_brems"]:
            sig, cdf = t["br"][d["Z"]]
            near = (self.x >= self.x0) & (self.x <= self.x1) & (gamma > 1 + p["photon_min_mc2"])
            if d["geometry"] == 1:
                near &= self.y.abs() <= self.yh
            k = near.nonzero()[:, 0]
            if len(k):
                a = self.words(k, n, 0)
                # no test passes above the largest probability of the table
                c = _uni53(a[0], a[1]) <= -math.expm1(-self.K * float(sig.max())) * (1 + 1e-9)
                k, a = k[c], [v[c] for v in a]
                gk = gamma[k]
                i, w = _row(gk, p["gamma_min"], p["gamma_max"], p["n_E"])
                um = torch.sqrt(sum(v[k] ** 2 for v in u))
                P = -torch.expm1(-self.K * ((1 - w) * sig[i] + w * sig[i + 1]) * um / gk)
                c = (a[1].double() * 2.0 ** 32 + a[0].double()) * 2.0 ** -64 < P
                k, i, w, gk = k[c], i[c], w[c], gk[c]
                if len(k):
                    j, fr = _invert(cdf, i, i + 1, w, _uni53(a[2][c], a[3][c]))
                    s = torch.where(j < 0, 0.0, (j + fr) / (p["n_s"] - 1))
                    yc, ym = p["photon_min_mc2"] / gk, 1 - 1 / gk
                    self.recoil(k, gamma, yc * torch.exp(s * torch.log(ym / yc)) * gk)
        self.x = self.x + self.dt * u[0] / gamma
        if d["geometry"] == 1:
            self.y = self.y + self.dt * u[1] / gamma


def _pairs_exact(case, seed):
    d, n, steps = _run_dict(case, seed), case["n"], case["steps"]
    tabs = _tabs(False)
    m, p = Model(dict(d, init_dist=0), 1, tabs), tabs["p"]
    rec = _photons(case, seed)
    v = rec[:, :6].contiguous().view(torch.float32).double()
    ne, idm = rec[:, 6].long(), rec[:, 7].long() & 0xFFFFFFFF
    k = v[:, 2]
    out = torch.zeros(n, 7, dtype=torch.float64, device=CUDA)
    sig, cdf = tabs["bh"][d["Z"]]
    i, w = _row(k, 2.0, p["gamma_max"], p["n_E"])
    lam = m.K * ((1 - w) * sig[i] + w * sig[i + 1])
    pos = v[:, 0] + v[:, 3] * m.dt
    first = torch.where((pos >= m.x0) & (pos <= m.x1), 1, 1 << 40)         # steps from the emission to the target
    first = torch.where((pos < m.x0) & (v[:, 3] > 0), torch.ceil((m.x0 - v[:, 0]) / (v[:, 3] * m.dt)).long(), first)
    live = ((k > 2) & (ne + first < steps)).nonzero()[:, 0]
    def convert(r, at, R):
        j, fr = _invert(cdf, i[r], i[r] + 1, w[r], R)
        x = 1 / k[r] + torch.where(j < 0, 0.0, (j + fr) / (p["n_s"] - 1)) * (1 - 2 / k[r])
        xe = v[r, 0] + v[r, 3] * ((at - ne[r]).double() * m.dt)
        out[r] = torch.stack([xe, 0 * xe, k[r] - x * k[r], x * k[r], v[r, 3], v[r, 4], v[r, 5]], 1)
    inside = lambda r, at: ((q := v[r, 0] + v[r, 3] * ((at - ne[r]).double() * m.dt)) >= m.x0) & (q <= m.x1)  # noqa: E731
    if case["method"] == "free":
        a = ne[live] + first[live]
        g = _philox(idm[live], 0 * a + m.run_id, a, 0x50000000 + ne[live], m.seed)
        at = a + torch.floor(-torch.log(_uni53(g[0], g[1])) / lam[live]).clamp(max=1e9).long()
        c = (at < steps) & inside(live, at)
        convert(live[c], at[c], _uni53(g[2][c], g[3][c]))
        return out
    P = -torch.expm1(-lam)
    for step in range(steps):
        r = live[ne[live] + first[live] <= step]
        if len(r):
            at = torch.full_like(r, step)
            gone = ~inside(r, at)
            g = _philox(idm[r], 0 * r + m.run_id, at, 0x40000000 + ne[r], m.seed)
            hit = ~gone & ((g[1].double() * 2.0 ** 32 + g[0].double()) * 2.0 ** -64 < P[r])
            convert(r[hit], at[hit], _uni53(g[2][hit], g[3][hit]))
            done = torch.zeros(n, dtype=torch.bool, device=CUDA)
            done[r[hit | gone]] = True
            live = live[~done[live]]
    return out


def _bw_tables(n_chi=64, lo=1e-2, hi=1e3, n_x=128):
    if "bw" not in _model:
        gx, gw = _gauss(16)
        chi = _log_grid(lo, hi, n_chi)
        s = (torch.arange(n_x - 1, device=CUDA)[:, None] + gx) / (n_x - 1)
        x = 0.5 * (1 - torch.cos(math.pi * s))
        ratio = x / (1 - x) + (1 - x) / x
        rows = []
        for c in chi:
            xi = 2 / (3 * c * x * (1 - x))
            ok = xi < 700
            q = torch.where(ok, xi, 700.0).reshape(-1)
            G = torch.where(ok, ratio * _bessel(2 / 3, q).view_as(xi) + _bessel(1 / 3, q, True).view_as(xi), 0.0)
            rows.append((G * 0.5 * math.pi * torch.sin(math.pi * s) * gw / (n_x - 1)).sum(1))
        total, cdf = _cumulated(torch.stack(rows))
        _model["bw"] = torch.log(total / (math.sqrt(3) * math.pi)) + 8 / (3 * chi), cdf, lo, hi, n_chi
    return _model["bw"]


def _bw_exact(case, seed):
    L, cdf, lo, hi, n_chi = _bw_tables()
    m = Model(dict(_run_dict(case, seed), init_dist=0), 1, _tabs(False))
    rec = _photons(case, seed)
    v = rec[:, :6].contiguous().view(torch.float32).double()
    ne, idm = rec[:, 6].long(), rec[:, 7].long() & 0xFFFFFFFF
    k, y0 = v[:, 2], v[:, 1]
    kv = [v[:, 2] * v[:, j] for j in (3, 4, 5)]
    kk = torch.sqrt(sum(q * q for q in kv))
    out = torch.zeros(len(k), 7, dtype=torch.float64, device=CUDA)
    g = _philox(idm, 0 * ne + m.run_id, ne, 0x60000000 + ne, m.seed)
    tau, open_ = -torch.log(_uni53(g[0], g[1])), k > 2
    flat = case["field"] != "gauss"
    for step in range(1, case["steps"]):
        r = (open_ & (ne < step)).nonzero()[:, 0]
        if not len(r):
            continue
        path = (step - ne[r]).double() * m.dt
        x, y = v[r, 0] + v[r, 3] * path, y0[r] + v[r, 4] * path
        E, B = m.fields(x, y, step * m.dt)
        chi = m.chi([q[r] for q in kv], kk[r], E, B, rest=0.0)
        i, w = _row(chi, lo, hi, n_chi)
        T = torch.exp((1 - w) * L[i] + w * L[i + 1] - 8 / (3 * torch.where(chi < hi, chi, hi)))
        tau[r] -= ALPHA * m.ES * m.dt * torch.where(chi >= lo, T, 0.0) / k[r]
        c = tau[r] <= 0
        q = r[c]
        if len(q):
            g = _philox(idm[q], 0 * q + m.run_id, 0 * q + step, 0x70000000 + ne[q], m.seed)
            j, fr = _invert(cdf, i[c], i[c] + 1, w[c], _uni53(g[0], g[1]))
            f = 0.5 * (1 - torch.cos(math.pi * (j + fr).clamp(min=0.0) / (cdf.shape[1] - 1)))
            out[q] = torch.stack([x[c], 0 * x[c] if flat else y[c], k[q] - f * k[q], f * k[q], v[q, 3], v[q, 4], v[q, 5]], 1)
            open_[q] = False
    return out


def exact(case, seed):
    f = case["family"]
    if f == "bh":
        return dict(values=_pairs_exact(case, seed), words=None, counts=None)
    if f == "bw":
        return dict(values=_bw_exact(case, seed), words=None, counts=None)
    steps = case.get("steps", 0) + case.get("before", 0)
    calm = (f == "job" and case["brems"] == "direct" and not case["box"] and case["field"] != "reflected" and
            (case["a0"] <= 60.0 or case["field"] == "gauss" and case["init"] == "rest" and steps <= 1000)) or (f == "bunch" and case["brems"] == "direct") or f == "stepwise"
    if not calm or steps > 2100 or case["n"] * steps > 2.2e9:
        return None
    with torch.no_grad():
        m = Model(_run_dict(case, seed), case["n"], _tabs(f != "bunch" and case.get("target") != "al" or f == "stepwise"))
        for k in range(steps):
            m.step(k)
    state = dict(x=m.x, tau=m.tau, ux=m.u[0], uy=m.u[1], uz=m.u[2])
    if case.get("field") == "gauss":
        state["y"] = m.y
    return dict(state=state)
