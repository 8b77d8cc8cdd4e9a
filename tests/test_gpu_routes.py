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
