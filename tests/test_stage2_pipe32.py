"""The 32-bit stage 2 (int32 and float32 intermediates) at the sizes where it
can go wrong: every warp split and two DMs per warp, ragged last groups, tiles
cut by the series' end, staged rows so long that fewer stages or a shorter
tile fit. int32 series equal the oracle bit for bit; float series lie within
the first-order rounding bound of their sums (oracle.normalise)."""
import numpy as np
import pytest

import synth
from oracle import dedisp as O
from oracle import normalise as NM
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# (group, ndm, nsamp, dm_max, tsamp): splits 4, 2 and 1, one and two DMs per warp
SHAPES = [(1, 2, 1, 30.0, 256e-6), (3, 7, 1023, 60.0, 256e-6), (7, 20, 1025, 60.0, 256e-6),
          (8, 17, 2048, 60.0, 256e-6), (14, 29, 1500, 60.0, 256e-6), (15, 31, 700, 60.0, 256e-6),
          (16, 16, 3000, 60.0, 256e-6), (17, 35, 513, 60.0, 256e-6), (32, 70, 1100, 60.0, 256e-6)]
# delay spreads (hundreds of samples) within a group that leave three, two and one stage of 1024 outputs, one of
# 512, and (groups of 32) one of 256
LONG = [(2, 2, 600, 2.0, 60.0), (2, 2, 600, 2.0, 200.0), (2, 2, 600, 2.0, 350.0), (2, 2, 600, 2.0, 570.0),
        (17, 17, 600, 2.0, 560.0), (32, 32, 600, 2.0, 572.6)]


def _series(tx, interm, norm, group, ndm, nsamp, dm_max, tsamp, seed):
    wl = synth.tiny_workload(nchan=32, nsub=4, ndm=ndm, nsamp=nsamp, dm_max=dm_max, widths=(1, 2, 4), tsamp=tsamp,
                             group=group)
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, wl.nsub, wl.widths, wl.nsamp, group=group, interm=interm, norm=norm,
                   output="series", tile_split2=1)
    X = synth.make_spectrum(wl, plan.overlap + nsamp, seed=seed)
    beam = tx.Beam(plan)
    beam.prime(torch.from_numpy(np.ascontiguousarray(X[:, :plan.overlap])).cuda())
    out = tx.execute(plan, beam, torch.from_numpy(np.ascontiguousarray(X[:, plan.overlap:])).cuda().reshape(-1))
    torch.cuda.synchronize()
    op = O.SubbandPlan(wl.freqs_mhz, wl.tsamp_s, wl.dms, wl.nsub, group, wl.widths)
    return tx.series_view(plan, out).cpu().numpy(), X, op, plan


def _tsamp(rows):
    """Sampling time giving two DMs of a group `rows` hundred samples of delay between them in the lowest sub-band."""
    wl = synth.tiny_workload(nchan=32, nsub=4, ndm=2, dm_max=2.0)
    f = wl.freqs_mhz
    return synth.sky_delay_samples(2.0, f[7], f[-1], 1.0) / (100.0 * rows)


@pytest.mark.parametrize("shape", SHAPES + LONG)
def test_int32_series_equal_the_oracle(tx, shape):  # noqa: F811
    group, ndm, nsamp, dm_max, ts = shape
    ts = ts if ts < 1.0 else _tsamp(ts)
    got, X, op, _ = _series(tx, "i32", "none", group, ndm, nsamp, dm_max, ts, 3)
    assert np.array_equal(got, O.subband_dedisperse(X, op, nsamp + op.wmax - 1))


@pytest.mark.parametrize("shape", SHAPES + LONG[2:])
def test_float_series_within_the_rounding_bound(tx, shape):  # noqa: F811
    group, ndm, nsamp, dm_max, ts = shape
    ts = ts if ts < 1.0 else _tsamp(ts)
    got, X, op, plan = _series(tx, "f32", "unit", group, ndm, nsamp, dm_max, ts, 4)
    Xn = NM.normalised_stream(X, plan.overlap, nsamp, 1, "unit").astype(np.float64)
    n = nsamp + op.wmax - 1
    D = O.subband_dedisperse(Xn, op, n)
    bound = NM.sum_error_bound(O.subband_dedisperse(np.abs(Xn), op, n), op.m + op.nsub + 1)
    assert np.all(np.abs(got.astype(np.float64) - D) <= bound)
