"""Mean and variance of the float path's series to the precision of sums in
double, where the variance is far below the squared mean (10^-10 of it).

The data make every series constant but for one sample: all channels are high in
the carried samples and the first half of the block, low after, so the
normalised values that the series sum are equal, and one count in one channel is
the only spread. The beam's running statistics (weight 1: the block's own) give mu
and var as the library holds them; the exact ones come from the float32 series.

Bound. The values share a binade, so squares are multiples of one ulp^2 with 48
bits and a lane's (at most 32) sum exactly in 53 bits, as do sums of values. What
rounds, by u = 2^-53 of at most mu^2 (or mu) each time: 5 additions across a warp's
lanes, one per part of the tiles, the division; so the mean square and twice the
mean are off by 6 + parts each, the square of the mean and the difference by 1 more:
|var - exact| <= (3 (6 + parts) + 2) u mu^2, |mu - exact| <= (6 + parts) u |mu|."""
from fractions import Fraction

import numpy as np
import pytest

import synth
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

T, WMAX, NCHAN = 2046, 1024, 64      # the overlap of DM 0 is WMAX - 1 = T / 2


def _blocks(seed):
    rng = np.random.default_rng(seed)
    lo = rng.integers(60, 100, NCHAN)
    hi = lo + rng.integers(80, 120, NCHAN)
    late = np.arange(T)[None, :] >= T // 2
    b0 = np.where(late, hi[:, None], lo[:, None]).astype(np.uint8)
    b1 = np.where(late, lo[:, None], hi[:, None]).astype(np.uint8)
    b1[5, 100] += 1
    return b0, b1


def _run(tx, blocks, group, ndm, **kw):  # noqa: F811
    wl = synth.tiny_workload(nchan=NCHAN, nsub=8, ndm=ndm, nsamp=T, dm_max=0.0, widths=(1, 2, WMAX), group=group)
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, wl.nsub, wl.widths, T, group=group, norm="invvar", **kw)
    assert plan.overlap == T // 2
    beam = tx.Beam(plan)
    beam.prime(torch.zeros((NCHAN, plan.overlap), dtype=torch.uint8, device="cuda"))
    for b in blocks:
        out = tx.execute(plan, beam, torch.from_numpy(b).cuda())
    torch.cuda.synchronize()
    return plan, beam, out


# groups: one warp per DM and 32 values a lane, two warps and 16, four and 8, two DMs per warp
@pytest.mark.parametrize("group,split", [(16, 1), (8, 2), (4, 4), (20, 1)])
@pytest.mark.parametrize("seed", [6, 7, 14, 31])
def test_mean_and_variance(tx, seed, group, split):  # noqa: F811
    blocks, ndm = _blocks(seed), group + 1
    plan, _, out = _run(tx, blocks, group, ndm, output="series")
    D = tx.series_view(plan, out).cpu().numpy()[:, :T]
    plan, beam, _ = _run(tx, blocks, group, ndm, output="plane", stats="running", stats_lambda=1.0)
    got = np.frombuffer(beam.export(), dtype=np.uint8)[-16 * ndm:].view(np.float64).reshape(ndm, 2)
    parts = split * -(-(T + WMAX - 1) // (512 if group > 16 else 1024))
    u = Fraction(1, 2 ** 53)
    for d in range(ndm):
        assert len(np.unique(D[d])) <= 4 and np.ptp(np.frexp(D[d])[1]) == 0      # the bound's premise
        q = [Fraction(float(x)) for x in D[d]]
        mu = sum(q) / T
        var = sum((x - mu) ** 2 for x in q) / T
        assert 0 < var < mu * mu * Fraction(1, 10 ** 9)
        assert abs(Fraction(float(got[d, 0])) - mu) <= (6 + parts) * u * mu
        assert abs(Fraction(float(got[d, 1])) - var) <= (3 * (6 + parts) + 2) * u * mu * mu
