"""Failure detection on the FP64 path, without a fault: with the test hook on, the tensor-core sums of
(P|Q) and (P|ij) wait for a flag that nothing clears; with a 2 ms limit that wait runs out, the status
word is set (psq_check: PSQ_ERR_TIMEOUT) and the elements read NaN.  The next compute on the same
workspace matches the oracle; the classes without tensor-core sums never wait."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mask", [oracle.ALL, 8])
def test_fp64_wait_timeout_is_reported(mask):
    import torch
    import paper_2510_15204_gb300 as P
    ctx = P.Context(0)
    job = synth.h2_fp64(0)
    J = P.Job.from_synth(ctx, job, P.FP64)
    ws, out = J.alloc(mask)
    J.set_wait_limit(2 * 10 ** 6)
    J.test_stall(True)
    J.compute(mask, ws, out)
    with pytest.raises(P.PsqError) as e:
        J.check(mask, ws)
    assert e.value.status == 4  # PSQ_ERR_TIMEOUT
    torch.cuda.synchronize()  # the context still answers
    assert bool(torch.isnan(out["J2"]).any())
    J.test_stall(False)
    J.compute(mask, ws, out)  # (with the short limit: every wait is far below it)
    J.check(mask, ws)
    ref = oracle.compute(job, mask=mask)
    for i, k in enumerate(P.CLASSES):
        if (mask >> i) & 1:
            err = np.abs(out[k].cpu().numpy() - ref[k])
            assert np.all(err <= 1e-12 * np.maximum(np.abs(ref[k]), ref["abs" + k])), k


def test_fp64_without_tensor_core_sums_never_waits():
    import paper_2510_15204_gb300 as P
    J = P.Job.from_synth(P.Context(0), synth.h2_fp64(0), P.FP64)
    mask = P.S | P.T | P.V
    ws, out = J.alloc(mask)
    J.set_wait_limit(2 * 10 ** 6)
    J.test_stall(True)
    J.compute(mask, ws, out)
    J.check(mask, ws)
