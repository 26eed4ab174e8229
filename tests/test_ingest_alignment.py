"""Blocks landing in the ring at every alignment: lengths of every residue mod
16, channel counts that leave 16-, 4- and 1-byte reads, blocks that begin off
any word, several blocks so that the ring wraps, compact beams and batches, the
integer and the float path. Series equal the oracle (float: within the
rounding bound of the sums)."""
import numpy as np
import pytest

import synth
from oracle import dedisp as O
from oracle import normalise as NM
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(32, 1, "ft"), (32, 17, "tf"), (20, 130, "ft"), (20, 67, "tf"), (18, 255, "tf"), (18, 301, "ft"),
         (80, 1024, "tf"), (66, 516, "tf"), (21, 4111, "ft"), (21, 73, "tf")]


def _offset(x, off):
    """The bytes of x as a CUDA tensor that begins `off` bytes into its allocation."""
    buf = torch.empty(x.size + 64, dtype=torch.uint8, device="cuda")
    v = buf[off:off + x.size]
    v.copy_(torch.from_numpy(np.ascontiguousarray(x).reshape(-1)))
    return v


def _lay(x, layout):
    return x.T if layout == "tf" else x


@pytest.mark.parametrize("nchan,nsamp,layout", CASES)
@pytest.mark.parametrize("kind", ["full", "compact", "batch", "float"])
def test_series_at_every_alignment(tx, nchan, nsamp, layout, kind):  # noqa: F811
    wl = synth.tiny_workload(nchan=nchan, nsub=1, ndm=5, nsamp=nsamp, dm_max=30.0, widths=(1, 2, 3), group=2)
    norm = "unit" if kind == "float" else "none"
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, 1, wl.widths, nsamp, group=2, layout=layout, output="series",
                   norm=norm)
    op = O.SubbandPlan(wl.freqs_mhz, wl.tsamp_s, wl.dms, 1, 2, wl.widths)
    L, T, nb = plan.overlap, nsamp, 4
    X = synth.make_spectrum(wl, L + nb * T, seed=nchan + nsamp)
    beam = tx.Beam(plan, compact=kind == "compact")
    beam.prime(_offset(_lay(X[:, :L], layout), 3))
    batch = tx.Batch([plan], [beam], graph=False) if kind == "batch" else None
    for b in range(nb):
        blk = _offset(_lay(X[:, L + b * T:L + (b + 1) * T], layout), (0, 4, 1, 16)[b])
        out, _ = plan.alloc_out()
        if batch:
            batch.execute([blk], [(out, None)], batch.alloc_workspace())
        else:
            tx.execute(plan, beam, blk, out=out)
        got = tx.series_view(plan, out).cpu().numpy()
        if kind == "float":
            w = NM.normalised_stream(X, L, T, nb, "unit").astype(np.float64)[:, b * T:b * T + L + T]
            n = T + op.wmax - 1
            bound = NM.sum_error_bound(O.subband_dedisperse(np.abs(w), op, n), op.m + op.nsub + 1)
            assert np.all(np.abs(got - O.subband_dedisperse(w, op, n)) <= bound)
        else:
            assert np.array_equal(got, O.subband_dedisperse(X[:, b * T:b * T + L + T], op, T + op.wmax - 1))
