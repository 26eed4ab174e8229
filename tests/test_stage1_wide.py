"""Stage 1 of sub-bands of many channels (k_stage1_wide) at the sizes where it can go
wrong: each length of its tiles, residues and spreads of every kind, coarse DMs
that fill an item and one more, blocks of one sample, rings shorter than a
window, lengths that give the windows every phase, every form of the
intermediates, batches of unlike beams. uint16 and int32 series equal the
oracle bit for bit, FP16 its emulation."""
import numpy as np
import pytest

import synth
from oracle import dedisp as O
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(tx, m, nsub, ndm, dm_max, nsamp, interm, descending=False, group=2):
    wl = synth.tiny_workload(nchan=m * nsub, nsub=nsub, ndm=ndm, nsamp=nsamp, dm_max=dm_max, widths=(1, 2, 4, 8),
                             group=group, descending=descending)
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, nsub, wl.widths, nsamp, group=group, interm=interm, output="series")
    op = O.SubbandPlan(wl.freqs_mhz, wl.tsamp_s, wl.dms, nsub, group, wl.widths)
    X = synth.make_spectrum(wl, plan.overlap + 2 * nsamp, seed=m + nsamp)
    return wl, plan, op, X


def _want(X, op, plan, b):
    w = X[:, b * plan.nsamp:b * plan.nsamp + plan.overlap + plan.nsamp]
    if plan.interm != "f16":
        return O.subband_dedisperse(w, op, plan.series_len)
    return O.subband_dedisperse_f16(w, op, plan.series_len, slice(plan.overlap, plan.overlap + plan.nsamp))


# (channels per sub-band, sub-bands, DMs, dm_max, block, descending): 8, 4 and 2 words per lane
SHAPES = [(65, 2, 20, 60.0, 1, False), (70, 1, 140, 40.0, 2500, True), (96, 2, 70, 900.0, 1000, False),
          (125, 2, 66, 90.0, 1531, True), (128, 1, 130, 200.0, 777, False), (160, 1, 36, 60.0, 1111, False),
          (200, 1, 70, 300.0, 640, True), (257, 2, 40, 120.0, 333, False)]
# lengths of whole 16 samples and others (the tiling moved by 1 to 15), from 16 channels on (128 coarse DMs: two full items)
ROWS = [(16, 3, 20, 60.0, 1003, True), (17, 2, 140, 90.0, 2001, False), (24, 2, 40, 300.0, 1, False),
        (32, 2, 66, 60.0, 1538, True), (33, 2, 20, 60.0, 16, False), (33, 1, 256, 40.0, 2512, True),
        (40, 2, 70, 900.0, 1008, False),
        (64, 2, 66, 90.0, 1536, True), (64, 1, 130, 200.0, 784, False), (64, 2, 40, 120.0, 779, False),
        (125, 2, 66, 90.0, 1536, False), (160, 1, 36, 60.0, 1120, True), (257, 1, 40, 120.0, 336, False)]


@pytest.mark.parametrize("interm", ["u16", "i32"])
@pytest.mark.parametrize("shape", SHAPES + ROWS)
def test_series_equal_the_oracle(tx, shape, interm):  # noqa: F811
    wl, plan, op, X = _setup(tx, *shape[:5], interm, shape[5])
    L, T = plan.overlap, plan.nsamp
    beam = tx.Beam(plan)
    beam.prime(torch.from_numpy(np.ascontiguousarray(X[:, :L])).cuda())
    for b in range(2):
        blk = torch.from_numpy(np.ascontiguousarray(X[:, L + b * T:L + (b + 1) * T])).cuda().reshape(-1)
        got = tx.series_view(plan, tx.execute(plan, beam, blk)).cpu().numpy()
        assert np.array_equal(got, _want(X, op, plan, b)), b
    assert beam.failed() == 0


@pytest.mark.parametrize("m,nsamp", [(100, 900), (100, 912), (64, 912)])
def test_noalloc_equals_the_oracle(tx, m, nsamp):  # noqa: F811
    wl, plan, op, X = _setup(tx, m, 2, 20, 60.0, nsamp, "u16")
    n = plan.overlap + plan.nsamp
    ld = (n + 63) // 64 * 64
    x = torch.zeros((wl.nchan, ld), dtype=torch.uint8, device="cuda")
    x[:, :n] = torch.from_numpy(X[:, :n].copy()).cuda()
    series = torch.empty(plan.ndm * plan.series_len, dtype=torch.int32, device="cuda")
    tx.dedisperse_noalloc(plan, x, ld, series)
    assert np.array_equal(series.view(plan.ndm, -1).cpu().numpy(), O.subband_dedisperse(X[:, :n], op, plan.series_len))


def test_batch_of_unlike_beams(tx):  # noqa: F811
    """Beams of several shapes and forms, compact and full, beside narrow ones; rows of the plan and sorted rows."""
    made = [_setup(tx, *s) for s in [(96, 2, 30, 60.0, 900, "u16"), (125, 1, 40, 80.0, 1100, "u16"),
                                     (96, 1, 50, 30.0, 513, "f16"), (16, 4, 24, 60.0, 800, "u16"),
                                     (125, 2, 20, 50.0, 640, "f16"), (64, 2, 24, 60.0, 640, "u16"),
                                     (64, 2, 24, 60.0, 650, "u16"), (40, 2, 30, 70.0, 656, "f16")]]
    plans = [p for _, p, _, _ in made]
    beams = [tx.Beam(p, compact=i % 2 == 0) for i, p in enumerate(plans)]
    for (_, p, _, X), bm in zip(made, beams):
        bm.prime(torch.from_numpy(np.ascontiguousarray(X[:, :p.overlap])).cuda())
    batch = tx.Batch(plans, beams, graph=False)
    outs, ws = batch.alloc_outs(), batch.alloc_workspace()
    for b in range(2):
        blocks = [torch.from_numpy(np.ascontiguousarray(X[:, p.overlap + b * p.nsamp:p.overlap + (b + 1) * p.nsamp]))
                  .cuda().reshape(-1) for _, p, _, X in made]
        batch.execute(blocks, outs, ws)
        torch.cuda.synchronize()
        for (_, p, op, X), (o, _) in zip(made, outs):
            assert np.array_equal(tx.series_view(p, o).cpu().numpy(), _want(X, op, p, b)), (b, p.nchan)
