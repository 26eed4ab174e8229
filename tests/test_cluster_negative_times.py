"""Clustering of records with times on both sides of zero (a caller that counts from
the block's start has the carried tail at negative times) and at the ends of the
type. Canonical order is that of the record's bits, negative times last in their DM;
neighbours, and so the clusters, are those of the signed times: order and labels equal
the oracle's DBSCAN of the points in that order."""
import numpy as np
import pytest

import synth
from oracle import cluster as CL
from test_cluster import gpu_cluster, make_plan, records, tx  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(tx, plan, wl, d, t, r_ms, k):  # noqa: F811
    d, t = np.asarray(d, dtype=np.int64), np.asarray(t, dtype=np.int64)
    rec = records(d, t, np.zeros(d.size), np.linspace(6, 9, d.size))
    _, labels, order = gpu_cluster(tx, plan, rec, r_ms, k)
    want = np.lexsort((t & 0xFFFFFFFF, d))
    assert np.array_equal(order, want)
    y = t[want].astype(np.float64) * (wl.tsamp_s * 1e3)
    ref, core = CL.dbscan(plan.delay_table()[d[want]], y, r_ms, k)
    assert np.array_equal(labels, ref)
    return ref, core


@pytest.mark.parametrize("r_samples", [1.0, 4.0, 10.0, 2.5])
@pytest.mark.parametrize("k", [0, 3])
def test_times_around_zero(tx, r_samples, k):  # noqa: F811
    wl = synth.tiny_workload(nchan=64, nsub=8, ndm=40, nsamp=4000, dm_max=12.0)
    plan = make_plan(tx, wl)
    rng = np.random.default_rng(int(10 * r_samples) + k)
    key = np.array(sorted({(int(a), int(b)) for a, b in zip(rng.integers(0, 40, 1500), np.round(rng.normal(0, 40, 1500)))}))
    rng.shuffle(key)
    _check(tx, plan, wl, key[:, 0], key[:, 1], r_samples * wl.tsamp_s * 1e3, k)


def test_one_row_through_zero(tx):  # noqa: F811
    """A row that is one cluster, its run of negative times after that of the others; a gap, a repeated record."""
    wl = synth.tiny_workload(nchan=64, nsub=8, ndm=40, nsamp=4000, dm_max=12.0)
    plan = make_plan(tx, wl)
    t = np.r_[np.arange(-30, 31, 2), -1, -1, 100, 102, 104]
    ref, core = _check(tx, plan, wl, np.full(t.size, 7), t, 3.0 * wl.tsamp_s * 1e3, 1)
    assert len(set(ref[core])) == 2


def test_ends_of_the_type(tx):  # noqa: F811
    wl = synth.tiny_workload(nchan=64, nsub=8, ndm=40, nsamp=4000, dm_max=12.0)
    plan = make_plan(tx, wl)
    t = np.r_[2 ** 31 - 1 - np.arange(0, 20, 2), -2 ** 31 + np.arange(0, 20, 2), np.arange(-6, 7, 2)]
    d = np.r_[np.arange(10) % 3, np.arange(10) % 3, np.arange(7) % 3]
    for r in (2.0, 5.0, 9.5):
        _check(tx, plan, wl, d, t, r * wl.tsamp_s * 1e3, 1)
