"""Failure handling that needs no GPU fault: particles whose momenta are not finite.

The caller's buffers (or arithmetic that overflowed) can hold a NaN or infinite momentum.
Every step kernel checks the state it loads at a launch boundary: such a particle is removed
(x = NaN, momenta zeroed), counted once in N_NONFINITE and N_KILLED with the steps it was
alive, and takes no further part; the other particles are untouched.  The bad values are
planted on the host, in the caller's buffers.
"""
import numpy as np
import pytest

import paper_1612_07592_gb300 as pe
from paper_1612_07592_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TP = dict(W.tables_small(), n_eta=48, n_y=48, n_E=48, n_s=48)
BAD = {5: ("ux", float("nan")), 17: ("uz", float("inf")), 300: ("uy", float("-inf")), 301: ("ux", float("nan"))}


@pytest.mark.parametrize("precision,launch", [(pe.PE_F32, {}), (pe.PE_F32, dict(steps_per_launch=1)),
                                              (pe.PE_F32, dict(steps_per_launch=50, block=128)),
                                              (pe.PE_F64, {}), (pe.PE_F64, dict(steps_per_launch=40))])
def test_nonfinite_momenta_removed_and_counted(precision, launch):
    import torch
    run = W.base_run(a0=270.0, init_dist=1, T_mev=1.0, seed=31, **W.AU)
    tables = pe.pe_create_tables(TP, (13.0, 79.0))
    n, steps = 1001, 120
    clean = pe.Run(tables, pe.run_params(precision=precision, **run), n, events=True)
    bad = pe.Run(tables, pe.run_params(precision=precision, **run), n, events=True)
    torch.cuda.synchronize()
    for i, (name, v) in BAD.items():
        getattr(bad, name)[i] = v
    pe.pe_step_ex([clean.handle], steps, **launch)
    pe.pe_step_ex([bad.handle], steps, **launch)
    sc, sb = clean.state(), bad.state()
    tb = bad.tally_out()
    tc = clean.tally_out()
    ids = np.array(sorted(BAD))
    keep = np.setdiff1d(np.arange(n), ids)
    np.testing.assert_array_equal(sb[keep], sc[keep])
    np.testing.assert_array_equal(bad.event_words()[keep], clean.event_words()[keep])
    assert np.isnan(sb[ids, 0]).all() and (sb[ids, 2:5] == 0).all()
    assert tb.tally[pe.T["N_NONFINITE"]] == len(BAD)
    assert tb.tally[pe.T["N_KILLED"]] == len(BAD) + tc.tally[pe.T["N_KILLED"]]
    assert tb.tally[pe.T["KILLED_STEPS"]] == tc.tally[pe.T["KILLED_STEPS"]]   # removed before step 0
    assert tb.live_particle_steps == tc.live_particle_steps - len(BAD) * steps
    # counted once: stepping on finds them removed
    pe.pe_step_ex([bad.handle], 10, **launch)
    assert bad.tally_out().tally[pe.T["N_NONFINITE"]] == len(BAD)
    clean.close()
    bad.close()
    pe.pe_destroy_tables(tables)


@pytest.mark.parametrize("precision,launch", [(pe.PE_F32, dict(steps_per_launch=1)), (pe.PE_F32, dict(steps_per_launch=3)),
                                              (pe.PE_F32, {}), (pe.PE_F64, {})])
def test_removed_electron_keeps_its_event_word(precision, launch):
    """An electron whose momentum turns non-finite after some emissions is removed with the event word it has (both
    electrons of a pair, either of them, and the odd last one), whatever the launch shape."""
    import torch
    run = W.base_run(a0=500.0, init_dist=1, seed=3, slab_x0_m=0.1e-6, slab_thick_m=0.7e-6, **W.AU)
    tables = pe.pe_create_tables(TP, (13.0, 79.0))
    n = 2001
    clean = pe.Run(tables, pe.run_params(precision=precision, **run), n, events=True)
    bad = pe.Run(tables, pe.run_params(precision=precision, **run), n, events=True)
    for r in (clean, bad):
        pe.pe_step_ex([r.handle], 110, **launch)
    words = bad.event_words()
    np.testing.assert_array_equal(words, clean.event_words())
    emitted = np.flatnonzero(words)
    assert len(emitted) > 20
    ids = np.unique(np.concatenate([emitted[::2], emitted[:6] ^ 1, [n - 1]]))
    ids = ids[ids < n]
    bad.uy[torch.from_numpy(ids).to(bad.uy.device)] = float("nan")
    for r in (clean, bad):
        pe.pe_step_ex([r.handle], 8, **launch)
    np.testing.assert_array_equal(bad.event_words()[ids], words[ids])
    keep = np.setdiff1d(np.arange(n), ids)
    np.testing.assert_array_equal(bad.event_words()[keep], clean.event_words()[keep])
    np.testing.assert_array_equal(bad.state()[keep], clean.state()[keep])
    assert bad.tally_out().tally[pe.T["N_NONFINITE"]] == len(ids)
    clean.close()
    bad.close()
    pe.pe_destroy_tables(tables)


@pytest.mark.parametrize("method", [pe.PE_BREMS_DIRECT, pe.PE_BREMS_NULL])
@pytest.mark.parametrize("precision,dense,launch", [(pe.PE_F32, False, {}), (pe.PE_F32, False, dict(steps_per_launch=20)),
                                                    (pe.PE_F32, True, {}), (pe.PE_F64, False, {})])
def test_removed_electron_takes_no_part_in_constant_fields(precision, dense, launch, method):
    """Electrons leave the box at different times while their partners in a pair go on: the removed ones emit nothing,
    keep their event words and are not counted (the fields of PE_CONST do not depend on the position).  dense: a target in
    which the lanes wait for one another's emissions.  The field lies along x (electrons leave along it) and every eta,
    u_perp B / E_S, is above the table, so N_ETA_ABOVE counts the steps of the live electrons."""
    tables = pe.pe_create_tables(dict(TP, eta_min=1e-6, eta_max=1e-5), (13.0, 79.0))
    target = dict(Z=79.0, charge_state=79.0, ne_over_nc=4177.0 * (50.0 if dense else 0.02))
    run = W.base_run(geometry=pe.PE_CONST, B_const=(2000.0, 0.0, 0.0), init_dist=1, seed=5, slab_x0_m=0.1e-6,
                     slab_thick_m=0.7e-6, box_enable=1, box_x_m=(0.0, 0.9e-6), brems_method=method, **target)
    n, steps = 3001, 60
    r = pe.Run(tables, pe.run_params(precision=precision, **run), n, events=True)
    x, words, emissions = np.zeros(n), np.zeros(n, np.uint64), 0
    for _ in range(4):
        pe.pe_step_ex([r.handle], steps, **launch)
        gone = np.isnan(x)
        w = r.event_words()
        np.testing.assert_array_equal(w[gone], words[gone])
        x, words = r.state()[:, 0], w
        t = r.tally_out()
        assert t.tally[pe.T["N_ETA_ABOVE"]] == t.live_particle_steps
        emissions = sum(int(t.tally[pe.T[k]]) for k in ("N_NCS_STORED", "N_NCS_BELOW", "N_BR_STORED", "N_BR_BELOW"))
        assert emissions == int((words & np.uint64(0xFFFF)).sum() + ((words >> np.uint64(16)) & np.uint64(0xFFFF)).sum())
        assert np.isfinite(r.photon_records()["x"]).all()
    assert emissions > 500 and 0 < np.isnan(x).sum()
    r.close()
    pe.pe_destroy_tables(tables)


@pytest.mark.parametrize("n,calls", [(70, (400,)), (70, (100, 300)), (70, (1,) * 400)])
def test_momenta_that_overflow_within_a_call(n, calls):
    """An FP64 run alone looks for non-finite momenta before every step, however many steps a call does: electrons that a
    huge constant field drives beyond the largest double are removed at that step and counted in that call."""
    E, dt = 1e307, 0.01 * 2 * np.pi
    tables = pe.pe_create_tables(TP, (13.0, 79.0))
    run = W.base_run(geometry=pe.PE_CONST, E_const=(E, 0.0, 0.0), enable_ncs=0, enable_brems=0, **W.AU)
    r = pe.Run(tables, pe.run_params(precision=pe.PE_F64, **run), n, events=True)
    for k in calls:
        pe.pe_step([r.handle], k)
    u, alive = 0.0, 0
    with np.errstate(over="ignore"):
        while np.isfinite(u):                       # two half kicks a step; the first steps to end beyond the range
            u = (u - 0.5 * dt * E) - 0.5 * dt * E
            alive += 1
    assert 10 < alive < 390
    t = r.tally_out()
    assert t.tally[pe.T["N_NONFINITE"]] == t.tally[pe.T["N_KILLED"]] == n
    assert t.tally[pe.T["KILLED_STEPS"]] == n * alive
    s = r.state()
    assert np.isnan(s[:, 0]).all() and (s[:, 2:5] == 0).all()
    r.close()
    pe.pe_destroy_tables(tables)
