"""The float path's stage 1 (a warp sums four coarse DMs, sharing equal delays) at
the sizes where it can go wrong: one channel, odd and large sub-bands, few and
many coarse DMs (every task shape), descending bands, block lengths that give
the ring every phase, equal and widely different delays. The series lie within
the first-order rounding bound of their sums (oracle.normalise)."""
import numpy as np
import pytest

import synth
from oracle import dedisp as O
from oracle import normalise as NM
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# (channels per sub-band, sub-bands, coarse DMs, dm_max, block length, descending)
@pytest.mark.parametrize("m,nsub,nk,dm_max,nsamp,descending", [
    (1, 3, 2, 30.0, 1, False), (2, 2, 5, 2000.0, 257, True), (3, 2, 10, 60.0, 1001, False),
    (16, 2, 17, 20.0, 1002, True), (17, 2, 25, 40.0, 1003, False), (31, 1, 40, 300.0, 512, False),
    (64, 2, 50, 25.0, 900, True), (125, 1, 64, 60.0, 640, False), (257, 1, 130, 90.0, 300, True),
    (8, 2, 64, 5000.0, 700, False)])
def test_series_within_the_rounding_bound(tx, m, nsub, nk, dm_max, nsamp, descending):  # noqa: F811
    wl = synth.tiny_workload(nchan=m * nsub, nsub=nsub, ndm=2 * nk, nsamp=nsamp, dm_max=dm_max, widths=(1, 3),
                             group=2, descending=descending)
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, nsub, wl.widths, nsamp, group=2, norm="unit", output="series")
    L, blocks = plan.overlap, 3
    X = synth.make_spectrum(wl, L + blocks * nsamp, seed=m)
    beam = tx.Beam(plan)
    beam.prime(torch.from_numpy(np.ascontiguousarray(X[:, :L])).cuda())
    op = O.SubbandPlan(wl.freqs_mhz, wl.tsamp_s, wl.dms, nsub, 2, wl.widths)
    Xn = NM.normalised_stream(X, L, nsamp, blocks, "unit").astype(np.float64)
    for b in range(blocks):
        blk = np.ascontiguousarray(X[:, L + b * nsamp:L + (b + 1) * nsamp])
        got = tx.series_view(plan, tx.execute(plan, beam, torch.from_numpy(blk).cuda().reshape(-1))).cpu().numpy()
        win = Xn[:, b * nsamp:b * nsamp + L + nsamp]
        D = O.subband_dedisperse(win, op, nsamp + op.wmax - 1)
        bound = NM.sum_error_bound(O.subband_dedisperse(np.abs(win), op, nsamp + op.wmax - 1), op.m + op.nsub + 1)
        assert np.all(np.abs(got.astype(np.float64) - D) <= bound), (b, float(np.abs(got - D).max()))
