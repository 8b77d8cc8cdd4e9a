"""Launch shapes and sizes at which a step, a conversion or a diagnostic takes another path, each against the path it
stands beside (bit for bit) or the oracle."""
import numpy as np
import pytest

import paper_1612_07592_gb300 as pe
from paper_1612_07592_gb300 import workloads as W

pytestmark = pytest.mark.gpu
Z = (13.0, 79.0)


def small_tables(**kw):
    return pe.pe_create_tables(dict(W.tables_small(), **dict(dict(n_eta=48, n_y=48, n_E=48, n_s=48), **kw)), Z)


def outcome(r):
    t = r.tally_out()
    ph = r.photon_records()
    order = np.lexsort((ph["step"], ph["id_mech"]))
    return r.state(), r.event_words(), bytes(t.tally), bytes(t.hist), ph[order].tobytes()


def same(a, b):
    np.testing.assert_array_equal(a[0], b[0])
    np.testing.assert_array_equal(a[1], b[1])
    assert a[2:] == b[2:]


@pytest.mark.parametrize("n", [1, 31, 33, 700])
def test_f64_one_warp_tiles_equal_larger_ones_and_single_steps(n):
    """An FP64 run alone (tiles of one warp, all steps in one launch) equals tiles of 64 in launches of 7 steps."""
    lt = small_tables()
    run = W.base_run(a0=270.0, init_dist=1, seed=5, slab_x0_m=0.5e-6, **W.AU)
    outs = []
    for cfg in ({}, dict(block=64, steps_per_launch=7), dict(steps_per_launch=1)):
        r = pe.Run(lt, pe.run_params(precision=pe.PE_F64, **run), n, events=True)
        pe.pe_step_ex([r.handle], 260, **cfg)
        outs.append(outcome(r))
    for o in outs[1:]:
        same(o, outs[0])


def test_f64_tables_beyond_shared_memory():
    """Rate tables larger than shared memory: an FP64 run alone reads them in place (results close to the small
    set's: the tables are finer), and what is refused for them stays refused."""
    big = pe.pe_create_tables(dict(W.tables_small(), n_eta=4096, n_y=8, n_E=4096, n_s=8), tuple(float(z) for z in range(75, 81)))
    run = W.base_run(a0=270.0, seed=5, slab_x0_m=0.5e-6, **W.AU)
    r = pe.Run(big, pe.run_params(precision=pe.PE_F64, **run), 300)
    pe.pe_step([r.handle], 150)
    ref = pe.Run(small_tables(n_eta=512, n_E=512), pe.run_params(precision=pe.PE_F64, **run), 300)
    pe.pe_step([ref.handle], 150)
    a, b = r.state(), ref.state()
    np.testing.assert_allclose(a[:, 5], b[:, 5], rtol=1e-3)     # the rates differ by the interpolation of 512 rows
    with pytest.raises(pe.PeError):
        pe.pe_step_ex([r.handle], 10, steps_per_launch=5)


@pytest.mark.parametrize("n_E,n_z", [(512, 1), (2048, 2), (3500, 4), (3840, 6)])
def test_f64_rate_tables_of_every_size(n_E, n_z):
    """FP64 runs read the rate tables where they are: alone, in launches of 7 steps, in a batch and replayed from a graph they
    give the same results with tables of 12 to 192 KB."""
    lt = pe.pe_create_tables(dict(W.tables_small(), n_eta=1024, n_y=16, n_E=n_E, n_s=16), tuple(79.0 - k for k in range(n_z)))
    run = W.base_run(a0=270.0, init_dist=1, seed=5, slab_x0_m=0.1e-6, slab_thick_m=0.7e-6, **W.AU)
    n, steps, outs = 700, 126, []
    for how in ("alone", "launches", "batch", "graph"):
        r = pe.Run(lt, pe.run_params(precision=pe.PE_F64, **run), n, events=True)
        if how == "alone":
            pe.pe_step([r.handle], steps)
        elif how == "launches":
            pe.pe_step_ex([r.handle], steps, steps_per_launch=7)
        elif how == "batch":
            other = pe.Run(lt, pe.run_params(precision=pe.PE_F64, **dict(run, run_id=1)), 50)
            pe.pe_step([r.handle, other.handle], steps)
        else:
            g = pe.pe_graph_create([r.handle], steps // 2)
            pe.pe_graph_launch(g)
            pe.pe_graph_launch(g)
        outs.append(outcome(r))
        if how == "graph":
            pe.pe_graph_destroy(g)
    assert outs[0][1].any()
    for o in outs[1:]:
        same(o, outs[0])


# --------------------------------------------------------------------------- the paired FP32 step ----
@pytest.mark.parametrize("n_eta,n_E,n_z", [(48, 48, 2), (1024, 2048, 3), (4096, 4096, 7)])
def test_f32_rate_tables_of_every_size(n_eta, n_E, n_z):
    """The paired kernels copy h(eta) and the run's own row of sigma_Z: runs of several Z give the same results alone, in
    launches of one step and in a batch in which a CTA goes from one row to another."""
    Zs = (13.0, 79.0, 29.0, 47.0, 6.0, 22.0, 73.0)[:n_z]
    lt = pe.pe_create_tables(dict(W.tables_small(), n_eta=n_eta, n_y=16, n_E=n_E, n_s=16), Zs)
    kw = dict(a0=400.0, init_dist=1, slab_x0_m=0.1e-6, slab_thick_m=0.7e-6, dt_over_T=0.02, charge_state=6.0, ne_over_nc=4000.0)

    def runs():
        return [pe.Run(lt, pe.run_params(precision=pe.PE_F32, **W.base_run(**dict(kw, Z=Zs[k % n_z], seed=k, run_id=k))),
                       3_001, events=True) for k in range(5)]
    alone, one, batch = runs(), runs(), runs()
    for r in alone:
        pe.pe_step([r.handle], 90)
    for r in one:
        pe.pe_step_ex([r.handle], 90, steps_per_launch=1)
    pe.pe_step_ex([r.handle for r in batch], 90, ctas_per_sm=1, block=64)
    assert sum(int(r.tally_out().tally[pe.T["N_BR_STORED"]]) for r in alone) > 0
    for a, b, c in zip(alone, one, batch):
        same(outcome(b), outcome(a))
        same(outcome(c), outcome(a))


@pytest.mark.parametrize("n", [1, 2, 63, 257, 5_000, 200_003])
@pytest.mark.parametrize("kind", ["plane", "plane-null-box"])
def test_one_step_launches_queue_their_emissions(n, kind):
    """Launches of one step (an emission waits in its warp's queue) equal launches of many."""
    lt = small_tables()
    kw = dict(brems_method=pe.PE_BREMS_NULL, box_enable=1, box_x_m=(0.0, 0.9e-6)) if kind != "plane" else {}
    run = W.base_run(a0=500.0, init_dist=1, seed=n, slab_x0_m=0.1e-6, slab_thick_m=0.7e-6, **kw, **W.AU)
    outs = []
    for cfg in (dict(steps_per_launch=1), dict(steps_per_launch=110), dict(steps_per_launch=3)):
        r = pe.Run(lt, pe.run_params(precision=pe.PE_F32, **run), n, capacity=1 << 21, events=True)
        pe.pe_step_ex([r.handle], 110, **cfg)
        outs.append(outcome(r))
    for o in outs[1:]:
        same(o, outs[0])


@pytest.mark.parametrize("n", [5, 3_001])
def test_held_emissions_equal_those_taken_at_once(n):
    """The bunch in Au at dt = T waits for company with its emissions; in a batch with a thin target, or in launches of
    one step, it does not: the same electrons, photons and sums."""
    lt = small_tables()
    dense = dict(W.bunch(1000.0, "Au")["run"])
    thin = dict(W.bunch(500.0, "Al", dt_over_T=0.1)["run"], run_id=3)

    def bunch(run):
        return pe.Run(lt, pe.run_params(precision=pe.PE_F32, **run), n, capacity=1 << 18, events=True)
    alone, steps, mixed, other = bunch(dense), bunch(dense), bunch(dense), bunch(thin)
    pe.pe_step([alone.handle], 900)
    pe.pe_step_ex([steps.handle], 900, steps_per_launch=1)
    pe.pe_step([mixed.handle, other.handle], 900)
    ref = outcome(alone)
    assert ref[1].any()
    same(outcome(steps), ref)
    same(outcome(mixed), ref)


# ------------------------------------------------------------------- binning of the diagnostics ----
MEC2 = 0.51099895


def near_edges(rng, edges, n):
    """Values at the edges of a log grid, off by relative amounts of 1e-8 .. 1e-3 (and well inside the bins)."""
    d = 10.0 ** rng.uniform(-8, -3, n) * rng.choice([-1.0, 1.0], n)
    d[::7] = rng.uniform(0.01, 0.9, len(d[::7])) * (edges[1] / edges[0] - 1.0)
    return rng.choice(edges, n) * (1.0 + d)


@pytest.mark.parametrize("precision", [pe.PE_F32, pe.PE_F64])
@pytest.mark.parametrize("n,bins,lo,hi", [(1, 1, 0.01, 1e4), (4099, 200, 0.01, 1e4), (20_001, 4096, 1.0, 50.0),
                                          (4098, 64, 1e-9, 1e-3)])
def test_spectrum_bins_at_the_edges(precision, n, bins, lo, hi):
    """Electrons whose energies lie at the bin edges are counted as the FP64 formula counts them (values so near an
    edge that another logarithm could place them differently are left out)."""
    import torch
    rng = np.random.default_rng(n)
    lt = small_tables()
    r = pe.Run(lt, pe.run_params(precision=precision, **W.base_run()), n)
    e = near_edges(rng, np.exp(np.linspace(np.log(lo), np.log(hi), bins + 1)), n) / MEC2
    u = np.sqrt(e * (e + 2.0))
    u = u.astype(np.float32 if precision == pe.PE_F32 else np.float64)
    ek = (np.sqrt(1.0 + u.astype(np.float64) ** 2) - 1.0) * MEC2
    with np.errstate(divide="ignore"):
        pos = (np.log(ek) - np.log(lo)) * (bins / (np.log(hi) - np.log(lo)))
    u[np.abs(pos - np.round(pos)) < 1e-9 * bins] = 0.0        # at rest: counted nowhere
    pos[u == 0.0] = -1.0
    r.ux.copy_(torch.from_numpy(u))
    r.uy.zero_()
    r.uz.zero_()
    inside = pos[(pos >= 0) & (pos < bins)]
    want = np.bincount(np.floor(inside).astype(int), minlength=bins)
    np.testing.assert_array_equal(r.electron_spectrum(bins, lo, hi).astype(np.int64), want)


@pytest.mark.parametrize("n,nx,ne", [(1, 1, 1), (5003, 40, 32), (3001, 200_000, 4)])
def test_photon_map_bins_at_the_edges(n, nx, ne):
    """The same for the photon map: positions and energies at the bin edges."""
    import torch
    rng = np.random.default_rng(nx)
    lt = small_tables()
    r = pe.Run(lt, pe.run_params(precision=pe.PE_F32, **W.base_run()), 4, capacity=n)
    kl = 2.0 * np.pi / W.LAMBDA
    x_lo, x_hi, lo, hi = -1.5e-6, 8e-6, 0.511, 1e4
    x = (x_lo + (x_hi - x_lo) * (rng.integers(0, nx + 1, n) / nx + 10.0 ** rng.uniform(-9, -2, n) / nx)) * kl
    p = np.zeros((n, 8), dtype=np.float32)
    p[:, 0] = x
    p[:, 2] = near_edges(rng, np.exp(np.linspace(np.log(lo), np.log(hi), ne + 1)), n) / MEC2
    px = (p[:, 0].astype(np.float64) - x_lo * kl) * (nx / ((x_hi - x_lo) * kl))
    pe_ = (np.log(p[:, 2].astype(np.float64) * MEC2) - np.log(lo)) * (ne / (np.log(hi) - np.log(lo)))
    unsure = (np.abs(px - np.round(px)) < 1e-9 * nx) | (np.abs(pe_ - np.round(pe_)) < 1e-9 * ne)
    p[unsure, 2] = 0.0
    r.photons.copy_(torch.from_numpy(p.view(np.int32).reshape(-1)))
    r.tally[pe.T["N_PHOTONS"]] = n
    ok = ~unsure & (px >= 0) & (px < nx) & (pe_ >= 0) & (pe_ < ne)
    want = np.bincount(np.floor(px[ok]).astype(int) * ne + np.floor(pe_[ok]).astype(int), minlength=nx * ne)
    got = r.photon_map(nx, x_lo, x_hi, ne, lo, hi).astype(np.int64).reshape(-1)
    np.testing.assert_array_equal(got, want)


# ------------------------------------------------------------------------------------- the 1D PIC ----
@pytest.mark.parametrize("precision", [pe.PE_F32, pe.PE_F64])
@pytest.mark.parametrize("n_cells", [4, 255, 256, 511, 512, 1023, 1024, 1500, 4096])
def test_pic_fields_advect_by_one_cell_per_step(precision, n_cells):
    """Without charge the wave variants move one cell a step along +-x whatever the blocks of the update: a random
    grid, shifted, with the laser in front."""
    import torch
    lt = small_tables()
    L = n_cells * 0.01e-6
    run = W.base_run(a0=5.0, polarisation=1, geometry=pe.PE_PIC_1D, n_cells=n_cells, ne_over_nc=0.0,
                     slab_x0_m=0.3 * L, slab_thick_m=0.3 * L, **W.AL | dict(charge_state=11.0))
    r = pe.Run(lt, pe.run_params(precision=precision, **run), 3)
    rng = np.random.default_rng(n_cells)
    g = torch.from_numpy(rng.uniform(-1.0, 1.0, 6 * n_cells + 5)).to(r.grid.dtype)
    r.grid.copy_(g)
    steps = 3
    pe.pe_step([r.handle], steps)
    a, b = g.numpy(), r.grid.cpu().numpy()
    n = n_cells
    np.testing.assert_array_equal(a[:n], b[:n])                     # E_x: no current
    for v in range(4):
        old, new = a[n + v * (n + 1): n + (v + 1) * (n + 1)], b[n + v * (n + 1): n + (v + 1) * (n + 1)]
        if v in (0, 2):                                             # F+, G+
            np.testing.assert_array_equal(new[steps:], old[:-steps])
        else:
            np.testing.assert_array_equal(new[:-steps], old[steps:])
            np.testing.assert_array_equal(new[-steps:], 0.0)


@pytest.mark.parametrize("precision", [pe.PE_F32, pe.PE_F64])
@pytest.mark.parametrize("n,n_cells", [(1, 300), (33, 300), (5_001, 300), (700_001, 400)])
def test_pic_queue_splits(precision, n, n_cells):
    """Steps in one call and in calls of one step agree bit for bit (each step launches by itself and may start under the
    end of the one before), and a run of several tiles a warp counts every emission once: photons, counts and
    energies of the sums agree with the photon records."""
    if precision == pe.PE_F64 and n > 10_000:
        n = 20_001
    lt = small_tables()
    run = W.base_run(a0=300.0, init_dist=1, seed=n, geometry=pe.PE_PIC_1D, n_cells=n_cells, slab_x0_m=0.3e-6, **W.AU)
    outs = []
    for calls in ((160,), (1,) * 20 + (70, 70)):
        r = pe.Run(lt, pe.run_params(precision=precision, **run), n, capacity=1 << 22, events=n < 10_000)
        for k in calls:
            pe.pe_step([r.handle], k)
        t = r.tally_out()
        ph = r.photon_records()
        outs.append((r.state(), r.grid.cpu().numpy(), bytes(t.tally), bytes(t.hist),
                     ph[np.lexsort((ph["step"], ph["id_mech"]))].tobytes()))
        assert len(ph) == t.tally[pe.T["N_NCS_STORED"]] + t.tally[pe.T["N_BR_STORED"]]
        np.testing.assert_allclose(ph["energy"].astype(np.float64).sum(), t.e_ncs_stored + t.e_br_stored, rtol=1e-6)
        assert sum(t.hist[:2 * pe.HIST_E_BINS]) == len(ph)
    np.testing.assert_array_equal(outs[0][0], outs[1][0])
    np.testing.assert_array_equal(outs[0][1], outs[1][1])
    assert outs[0][2:] == outs[1][2:]


@pytest.mark.parametrize("precision,n_eta,n_z,n_E", [(pe.PE_F64, 1200, 7, 3550), (pe.PE_F32, 2800, 13, 3846)])
def test_pic_rate_tables_read_in_place(precision, n_eta, n_z, n_E):
    """Rate tables that leave no room for the warps' queues beside a grid of 400 cells are read in global memory: the same
    steps as on a grid of 300 cells, where they fit (nothing reaches the 300th), for a few electrons and for many tiles
    a warp."""
    lt = pe.pe_create_tables(dict(W.tables_small(), n_eta=n_eta, n_y=16, n_E=n_E, n_s=16), (79.0,) + tuple(range(60, 59 + n_z)))
    for n in (500, 130_001):
        outs = []
        for n_cells in (400, 300):
            run = W.base_run(a0=600.0, init_dist=1, seed=n, geometry=pe.PE_PIC_1D, n_cells=n_cells, slab_x0_m=0.3e-6, **W.AU)
            r = pe.Run(lt, pe.run_params(precision=precision, **run), n, events=True)
            pe.pe_step([r.handle], 120)
            outs.append(outcome(r))
        assert outs[0][1].any()
        same(outs[0], outs[1])
        t, ph, w = r.tally_out(), r.photon_records(), outs[0][1]
        stored, below = (t.tally[pe.T["N_NCS_" + k]] + t.tally[pe.T["N_BR_" + k]] for k in ("STORED", "BELOW"))
        assert len(ph) == stored == sum(t.hist[:2 * pe.HIST_E_BINS])
        assert int((w & np.uint64(0xFFFF)).sum() + ((w >> np.uint64(16)) & np.uint64(0xFFFF)).sum()) == stored + below
        np.testing.assert_allclose(ph["energy"].astype(np.float64).sum(), t.e_ncs_stored + t.e_br_stored, rtol=1e-6)


# ------------------------------------------------------------------------- pair production queues ----
@pytest.mark.parametrize("n", [1, 33, 3_000, 40_001])
@pytest.mark.parametrize("process", ["bh-direct", "bh-free", "bw-f32", "bw-f64"])
def test_transport_of_parts_equals_the_whole(process, n):
    """Photons taken in one call and in two calls of uneven parts convert alike (shares, rounds and queues differ)."""
    lt = small_tables()
    kl = 2.0 * np.pi / W.LAMBDA
    if process.startswith("bh"):
        run = dict(W.bunch(1000.0, "Au", thickness_m=1e-3)["run"])
        ph = W.synthetic_photons(n, 5, (0.0, 1500.0), (2.0, 4000.0), (0, 300), theta_max=0.3)
    else:
        run = W.base_run(a0=400.0, reflect_r=1.0, mirror_x_m=3e-6, seed=5, **W.AU)
        ph = W.synthetic_photons(n, 5, (1e-6 * kl, 4e-6 * kl), (100.0, 20000.0), (0, 300), theta_max=0.6)
    bw = pe.pe_bw_tables_create()
    r = pe.Run(lt, pe.run_params(precision=pe.PE_F64 if process == "bw-f64" else pe.PE_F32, **run), 16)
    pe.pe_step([r.handle], 700)

    def go(p):
        if process.startswith("bw"):
            return r.bw_transport(bw, photons=p)
        return r.pair_transport(photons=p, method=int(process == "bh-free"))
    cut = n // 3
    whole, parts = go(ph), [go(ph[:cut]), go(ph[cut:])] if cut else [go(ph)]
    for k, p in enumerate(parts[1:]):
        p[0]["photon"] += cut
    got = np.concatenate([p[0] for p in parts])
    key = lambda a: a[np.argsort(a["photon"])].tobytes()  # noqa: E731
    assert key(got) == key(whole[0]) and sum(p[1] for p in parts) == whole[1]
    for w in ("N_ENTERED", "N_K_ABOVE", "N_TESTS"):
        assert sum(int(p[2][pe.PT[w]]) for p in parts) == int(whole[2][pe.PT[w]])
    for w in ("E_PAIRS", "E_POSITRONS"):
        val = lambda t: int(t[pe.PT[w]]) + (int(t[pe.PT[w] + 1]) << 64)  # noqa: E731
        assert sum(val(p[2]) for p in parts) == val(whole[2])
