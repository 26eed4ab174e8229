"""The clustering's row index at the points where it can go wrong: radii that
are a whole number of samples (interval ends on the radius), several records
of one point, runs broken by gaps, many neighbours wanted, DM grids too fine
for it (the cell grid then) and just fine enough. Everything equals the
oracle's DBSCAN."""
import numpy as np
import pytest

import synth
from test_cluster import check, clustered_points, make_plan, records, tx  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _plan(tx, ndm, dm_max, tsamp=64e-6):  # noqa: F811
    wl = synth.tiny_workload(nchan=64, nsub=8, ndm=ndm, nsamp=4000, dm_max=dm_max, tsamp=tsamp)
    return wl, make_plan(tx, wl)


# radii in samples: whole ones, halves, next to whole ones
@pytest.mark.parametrize("r_samples", [1.0, 3.0, 10.0, 2.5, 7.0 * (1 + 1e-15), 7.0 * (1 - 1e-15)])
@pytest.mark.parametrize("k", [0, 2, 12])
def test_whole_sample_radii(tx, r_samples, k):  # noqa: F811
    wl, plan = _plan(tx, 40, 12.0)
    rec = clustered_points(np.random.default_rng(int(10 * r_samples) + k), wl.ndm, wl.nsamp, 25, 150, 200)
    check(tx, plan, rec, r_samples * wl.tsamp_s * 1e3, k)


def test_lattice_on_the_radius(tx):  # noqa: F811
    """Rows and times spaced by exactly the radius in time and by DMs of equal delay."""
    wl, plan = _plan(tx, 6, 0.0)          # every DM 0: all rows at one delay
    d, t = np.meshgrid(np.arange(6), np.arange(0, 3000, 5), indexing="ij")
    for r in (5.0, 4.999999, 10.0):
        check(tx, plan, records(d.ravel(), t.ravel(), np.zeros(d.size), np.linspace(6, 9, d.size)), r * 64e-3, 4)


def test_repeated_records(tx):  # noqa: F811
    wl, plan = _plan(tx, 30, 9.0)
    a = clustered_points(np.random.default_rng(5), wl.ndm, wl.nsamp, 10, 80, 60)
    rec = np.concatenate([a, a[::3], a[::3]])
    check(tx, plan, rec, 0.5, 3)


# DM trials within the radius: 300 (cells), 250 (rows)
@pytest.mark.parametrize("per_radius", [300, 250])
def test_fine_dm_grids(tx, per_radius):  # noqa: F811
    wl, plan = _plan(tx, 700, 10.0)
    step = float(np.diff(plan.delay_table())[0])
    rec = clustered_points(np.random.default_rng(per_radius), wl.ndm, wl.nsamp, 30, 60, 300)
    check(tx, plan, rec, per_radius * step, 2)
