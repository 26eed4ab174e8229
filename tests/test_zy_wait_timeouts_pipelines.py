"""Waits that give up in the pipelined kernels: stage 1 of wide sub-bands (one
beam and a batch), stage 1 of the float path, stage 2 of 32-bit intermediates.

As in the test of the other kernels (after which this file is collected) a
polling limit makes waits give up without any fault; here also a limit of one
poll, where some warps of a block pass and others do not. A warp goes on or
gives up as a whole, so that nothing is copied that was not announced and every
block returns: the call either reports TX_ERR_ABORTED and marks the beam, or
its results are exact, and after a reset they are exact again.
"""
import numpy as np
import pytest

import synth
from test_float_path import tx  # noqa: F401  (the built package)

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _setup(tx, interm):  # noqa: F811
    """32 channels per sub-band; a block of every kernel fills its stages several times."""
    wl = synth.tiny_workload(nchan=256, nsub=8, ndm=600, nsamp=60000, dm_max=60.0, widths=(1, 2, 4), group=2)
    plan = tx.Plan(wl.freqs_mhz, wl.tsamp_s, wl.dms, wl.nsub, wl.widths, wl.nsamp, group=2, interm=interm,
                   norm="unit" if interm == "f32" else "none", output="series")
    X = np.random.default_rng(7).integers(0, 256, size=(plan.nchan, plan.overlap + plan.nsamp), dtype=np.uint8)
    return plan, torch.from_numpy(np.ascontiguousarray(X[:, :plan.overlap])).cuda(), \
        np.ascontiguousarray(X[:, plan.overlap:])


def _primed(tx, plan, tail):  # noqa: F811
    beam = tx.Beam(plan)
    beam.prime(tail)
    return beam


@pytest.mark.parametrize("polls", [0, 1])
@pytest.mark.parametrize("interm", ["u16", "i32", "f32"])
def test_one_beam(tx, interm, polls):  # noqa: F811
    plan, tail, blk = _setup(tx, interm)
    ref = tx.execute(plan, _primed(tx, plan, tail), torch.from_numpy(blk).cuda())
    torch.cuda.synchronize()
    ref = ref.cpu().numpy()
    beam = _primed(tx, plan, tail)
    ws = plan.alloc_workspace()
    out, _ = plan.alloc_out()
    staging = torch.empty(plan.block_bytes, dtype=torch.uint8, device="cuda")
    h_out = np.zeros(plan.out_bytes, dtype=np.uint8)
    before = tx.wait_timeouts()
    old = tx.set_wait_polls(polls)
    try:
        tx.execute_host(plan, beam, blk, h_out, staging, out, None, ws)
        gave_up = False
    except tx.TxError as e:
        assert e.code == tx.TX_ERR_ABORTED
        gave_up = True
    finally:
        torch.cuda.synchronize()
        tx.set_wait_polls(old)
    assert gave_up or polls
    assert (beam.failed() > 0) == gave_up and (tx.wait_timeouts() > before) == gave_up
    if not gave_up:
        assert np.array_equal(h_out, ref)
    beam.reset()
    beam.prime(tail)
    tx.execute_host(plan, beam, blk, h_out, staging, out, None, ws)
    assert beam.failed() == 0 and np.array_equal(h_out, ref)


def test_every_beam_of_a_batch_is_marked(tx):  # noqa: F811
    plan, tail, blk = _setup(tx, "u16")
    beams = [_primed(tx, plan, tail) for _ in range(2)]
    batch = tx.Batch([plan, plan], beams, graph=False)
    ws, outs = batch.alloc_workspace(), batch.alloc_outs()
    d_blk = torch.from_numpy(blk).cuda()
    old = tx.set_wait_polls(0)
    try:
        batch.execute([d_blk, d_blk], outs, ws)
        with pytest.raises(tx.TxError) as e:
            batch.wait()
    finally:
        torch.cuda.synchronize()
        tx.set_wait_polls(old)
    assert e.value.code == tx.TX_ERR_ABORTED
    assert all(b.failed() > 0 for b in beams)
    for b in beams:
        b.reset()
        b.prime(tail)
    batch.execute([d_blk, d_blk], outs, ws)
    batch.wait()
    ref = tx.execute(plan, _primed(tx, plan, tail), d_blk)
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref) for o, _ in outs)
