"""Choices of a path whose wrong side costs 1.5 times and more, by the ratio of two calls
timed in turn on the same device (the best of nine; the limits lie between the two sides)."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
LN2 = float(np.log(2.0))


def _times(objs, calls, rounds=9):
    """Best seconds of each call, the calls taken in turn."""
    got = [[] for _ in calls]
    for k in range(rounds + 2):
        for i, (o, call) in enumerate(zip(objs, calls)):
            o.sync()
            t = time.perf_counter()
            call()
            o.sync()
            if k >= 2:
                got[i].append(time.perf_counter() - t)
    return [min(g) for g in got]


def _ensemble(n, nrep, taus, stencil, launch, resident):
    from paper_2212_07848_gb300.ensemble import Ensemble
    e = Ensemble([(n, n, -3.6 - 0.0002 * r, taus[r % len(taus)], 1e-6, LN2) for r in range(nrep)],
                 stencil=stencil, seed=3)
    e.set_resident(resident)
    e.set_launch(launch)
    e.init(1e-3)
    return e


@pytest.mark.parametrize("stencil", [4, 8])
@pytest.mark.parametrize("launch", ["LB_ENS_PER_STEP", "LB_ENS_PERSISTENT"])
def test_ensembles_of_mixed_rates(launch, stencil):
    """Every second replica at unit rates is no slower than none of them."""
    from paper_2212_07848_gb300 import abi
    es = [_ensemble(64, 304, taus, stencil, getattr(abi, launch), abi.LB_ENS_RESIDENT_OFF)
          for taus in ([0.9], [1.0, 0.9])]
    general, mixed = _times(es, [lambda e=e: e.step(64) for e in es])
    for e in es:
        e.close()
    assert mixed < 1.15 * general


@pytest.mark.parametrize("n,nrep", [(128, 8), (256, 16), (1024, 1)])
@pytest.mark.parametrize("launch", ["LB_ENS_PER_STEP", "LB_ENS_PERSISTENT"])
def test_default_bands_of_small_ensembles(launch, n, nrep):
    """The default height, and a height that is set, on ensembles that tall bands leave
    on a part of the SMs, against bands of 6 rows."""
    from paper_2212_07848_gb300 import abi
    es = [_ensemble(n, nrep, [1.0], 4, getattr(abi, launch), abi.LB_ENS_RESIDENT_OFF)
          for _ in range(3)]
    es[0].set_strip_height(6)
    es[2].set_strip_height(32)
    low, default, tall = _times(es, [lambda e=e: e.step(64) for e in es])
    for e in es:
        e.close()
    assert default < 1.4 * low and tall < 1.4 * low


def test_resident_ensembles_of_mixed_rates():
    """Replicas of both paths that fill the SMs once: not two half-empty launches."""
    from paper_2212_07848_gb300 import abi
    es = [_ensemble(64, 152, taus, 4, abi.LB_ENS_PER_STEP, abi.LB_ENS_RESIDENT_ON)
          for taus in ([0.9], [1.0, 0.9])]
    assert all(e.num_resident == 152 for e in es)
    general, mixed = _times(es, [lambda e=e: e.step(64) for e in es])
    for e in es:
        e.close()
    assert mixed < 1.25 * general


@pytest.mark.parametrize("nrep,taus", [(5, [1.0, 0.9]), (6, [0.9, 0.9, 1.0])])
def test_merged_residents_keep_their_bits(nrep, taus):
    from paper_2212_07848_gb300 import abi
    out = []
    for mode in (abi.LB_ENS_RESIDENT_ON, abi.LB_ENS_RESIDENT_OFF):
        e = _ensemble(32, nrep, taus, 8, abi.LB_ENS_PER_STEP, mode)
        e.sk_config(4, 4)
        e.step(13)
        e.sync()
        out.append([e.populations(r) for r in range(nrep)])
        e.close()
    assert all(np.array_equal(a, b) for a, b in zip(*out))


def test_many_small_residents_at_general_rates():
    """32^2 replicas of the general path, two CTAs an SM: less than 1.4 times the unit
    path's time (one CTA an SM: 1.6)."""
    from paper_2212_07848_gb300 import abi
    es = [_ensemble(32, 2000, [tau], 4, abi.LB_ENS_PER_STEP, abi.LB_ENS_RESIDENT_ON)
          for tau in (1.0, 0.9)]
    unit, general = _times(es, [lambda e=e: e.step(64) for e in es])
    for e in es:
        e.close()
    assert general < 1.4 * unit


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_a_strip_height_leaves_the_automatic_layout(tau):
    """A height set on a lattice that runs in tiles by itself (strips of 32 rows: 9 times)."""
    from paper_2212_07848_gb300.lattice import Lattice
    gs = [Lattice(256, 256, -3.8, tau, 1e-6) for _ in range(2)]
    for g in gs:
        g.init(LN2, 5, 1e-3)
    gs[1].set_strip_height(32)
    default, tall = _times(gs, [lambda g=g: g.step(64) for g in gs])
    assert np.array_equal(*(g.download_state() for g in gs))
    for g in gs:
        g.close()
    assert tall < 1.3 * default


@pytest.mark.parametrize("box", [(32, 32, 32), (64, 32, 128), (32, 8, 256)])
def test_3d_shells_beyond_the_last_mode(box):
    """Bins that no mode falls into are 0 and cost nothing (a pass over the rows for each
    of 5000 took 2.5 times the read-out of the others and more)."""
    from paper_2212_07848_gb300.lattice3 import Lattice3
    g = Lattice3(*box, -6.0, 1.0, 1e-6)
    g.init(LN2, 5, 1e-3)
    g.sk_config(2, 2)
    g.sk_full()
    g.step(2)
    shells = int(np.ceil(np.sqrt(3.0) * max(box) / 2)) + 1
    some, n = g.structure_factor(shells)
    for nbins in (shells - 1, shells + 1, 4096, 5000):
        every, m = g.structure_factor(nbins)
        k = min(nbins, shells)
        assert m == n and np.array_equal(every[:k], some[:k]) and not every[k:].any()
    a, b = _times([g, g], [lambda k=k: [g.structure_factor(k) for _ in range(20)]
                           for k in (shells, 5000)])
    g.close()
    assert b < 1.4 * a
