"""Pinned host fields are read and written by the kernels where they are, others
through device memory: the same bits either way, whatever mix, offset or overlap
of arrays decides the route."""
import numpy as np
import pytest

from paper_1308_0653_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _pinned(shape, offset=0):
    import torch
    n = int(np.prod(shape))
    return torch.empty(n + offset, dtype=torch.float64, pin_memory=True).numpy()[offset:].reshape(shape)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("nr,nth", [(1, 3), (33, 5), (257, 130), (1000, 900)])
@pytest.mark.parametrize("kinds", ["ppppp", "ppqpp", "mpppp", "pp-p-", "shared"])
def test_same_bits_as_pageable(nr, nth, precision, kinds):
    import torch
    from paper_1308_0653_gb300 import dbm
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = W.explosion(nr, nth, nsteps=0, seed=nr, dt=1e-7)
    shape = (nth, nr)
    ref_in = [np.ascontiguousarray(w.fields[k], dtype=np.float64).reshape(shape).copy() for k in dbm.FIELDS]
    sim = dbm.Simulation(dict(w.params, precision=precision))
    dbm.dbm_init_state(sim.h, *ref_in)
    ref_f = sim.export_state()
    ref, ref_tot = [np.empty(shape) for _ in range(5)], np.zeros(4)
    dbm.dbm_moments(sim.h, *ref, totals=ref_tot)

    # p pinned, q pinned at an odd offset, m pageable, - not wanted
    make = {"p": lambda: _pinned(shape), "q": lambda: _pinned(shape, 3), "m": lambda: np.empty(shape)}
    if kinds == "shared":  # two outputs a row apart in one allocation
        block = _pinned((nth + 1, nr))
        arrs = [make["p"]() for _ in range(3)] + [block[:nth], block[1:]]
    else:
        arrs = [make.get(k, make["p"])() for k in kinds]
    if kinds != "shared":
        for a, r in zip(arrs, ref_in):
            a[...] = r
        dbm.dbm_init_state(sim.h, *arrs)
        got = sim.export_state()
        assert np.array_equal(got[0], ref_f[0]) and np.array_equal(got[1], ref_f[1])
    outs = [None if k == "-" else a for k, a in zip(kinds, arrs)] if kinds != "shared" else arrs
    for a in outs:
        if a is not None:
            a[...] = -7.0
    tot = np.zeros(4)
    dbm.dbm_moments(sim.h, *outs, totals=tot)
    if kinds == "shared":  # what the copies in their order leave in pageable arrays that overlap alike
        same = np.full((nth + 1, nr), -7.0)
        ref[3:] = [same[:nth], same[1:]]
        dbm.dbm_moments(sim.h, *ref)
    for a, r in zip(outs, ref):
        if a is not None:
            assert np.array_equal(a, r)
    # the totals' partial sums run over other blocks: nr nth terms of one sign or nearly
    scale = max(abs(ref_tot[0]), abs(ref_tot[3]))
    assert np.abs(tot - ref_tot).max() <= 2.0 * nr * nth * np.finfo(float).eps * scale
    bad = ref_in[3].copy()
    bad[0, 0] = -1.0
    arrs[3][...] = bad
    for k in (0, 1, 2, 4):
        arrs[k][...] = ref_in[k]
    if kinds != "shared":
        with pytest.raises(dbm.DbmError):
            dbm.dbm_init_state(sim.h, *arrs)
    sim.close()
