"""Planes, cubes and candidates of plans with int32 intermediates equal those of the
uint16 plan of the same shape bit for bit: their statistics come from the 32-bit
stage 2's own tile sums (four, two and one warp per DM, two DMs per warp)."""
import numpy as np
import pytest

import synth
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(tx, wl, interm, output, blocks):  # noqa: F811
    kw = dict(snr_threshold=0.5, max_cands=1 << 18) if output == "cands" else {}
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, wl.nsub, wl.widths, wl.nsamp, group=wl.group, interm=interm,
                   output=output, stats="running", stats_lambda=0.5, **kw)
    beam = tx.Beam(plan)
    res = []
    for b in blocks:
        r = tx.execute(plan, beam, b)
        torch.cuda.synchronize()
        if output == "cands":
            rec, n = tx.cands_view(plan, *r)
            assert 0 < n <= plan.max_cands
            res.append(np.sort(rec, order=["dm_index", "t"]).tobytes())
        else:
            res.append(r.cpu().numpy().tobytes())
    return res


@pytest.mark.parametrize("output", ["plane", "cube", "cands"])
@pytest.mark.parametrize("group", [3, 7, 8, 14, 15, 17, 32])
def test_equal_to_uint16(tx, group, output):  # noqa: F811
    wl = synth.tiny_workload(nchan=32, nsub=4, ndm=2 * group + 1, nsamp=2500, dm_max=60.0, group=group)
    rng = np.random.default_rng(group)
    blocks = [torch.from_numpy(rng.integers(0, 256, size=(wl.nchan, wl.nsamp), dtype=np.uint8)).cuda() for _ in range(2)]
    assert _run(tx, wl, "i32", output, blocks) == _run(tx, wl, "u16", output, blocks)
