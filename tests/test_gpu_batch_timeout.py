"""A copy wait that runs out in one problem of a fused batched launch ends the
block, which then leaves out its frames of other problems too: each problem
that misses frames has to say so, and one that misses none stays right."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu


def _setup(m, side, seed, npeaks=1, step=3):
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(m + 40, m, side, step, npeaks=npeaks, offset=-2, seed=seed)
    case = Case(spec, scan=scan, state="perturbed", seed=seed)
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    return case, p, tuple(torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha))


def _run(sets, stalled):
    """Statuses of a call with the stalled problem's waits running out, and the results."""
    from paper_2312_14907_gb300 import mpbp
    probs, states = [s[1] for s in sets], [s[2] for s in sets]
    probs[stalled].set_test_stall(True)
    outs = mpbp.loss_grad_batched(probs, states)
    status = []
    for p in probs:
        try:
            p.sync_status()
            status.append(0)
        except mpbp.MPBPError as e:
            status.append(e.status)
    probs[stalled].set_test_stall(False)
    return status, outs


def _check(case, got):
    f, gr, gu, ga = case.oracle_loss_grad()
    assert abs(got[0].item() - f) <= 1e-5 * abs(f)
    for a, b in zip(got[1:], (gr, gu, ga)):
        assert rel_l2(a.cpu().numpy(), b) <= 1e-4


def test_m128_problems_behind_a_timeout_report_it():
    from paper_2312_14907_gb300 import mpbp
    # one block per SM, runs of equal length over the problems' frames in turn
    sets = [_setup(128, side, i) for i, side in enumerate((7, 13, 1, 1, 13))]
    probs = [s[1] for s in sets]
    probs[0].set_batch_schedule(1, 0)
    n = [p.nframes for p in probs]
    base = np.concatenate([[0], np.cumsum(n)])
    grid, stalled = min(int(base[-1]), probs[0].info()["num_sms"]), 1
    owner = np.repeat(np.arange(len(n)), n)
    missed = set()
    for b in range(grid):
        run = owner[base[-1] * b // grid: base[-1] * (b + 1) // grid]
        at = np.flatnonzero(run == stalled)
        if at.size:
            missed.update(run[at[0]:].tolist())
    assert stalled in missed and len(missed) > 1 and len(missed) < len(n)
    status, outs = _run(sets, stalled)
    for k, s in enumerate(status):
        assert s == (5 if k in missed else 0), (k, status, sorted(missed))    # MPBP_ERR_TIMEOUT
    for k, (case, _, _) in enumerate(sets):
        if k not in missed:
            _check(case, outs[k])
    for (case, p, _), got in zip(sets, mpbp.loss_grad_batched(probs, [s[2] for s in sets])):
        _check(case, got)
        p.sync_status()


@pytest.mark.parametrize("m,side,blocks", [(32, 36, 32), (64, 20, 8)])
def test_small_frames_behind_a_timeout_report_it(m, side, blocks):
    from paper_2312_14907_gb300 import mpbp
    # grouped by problem, block b takes items b, b + grid, ...: with at least a
    # grid of frames in the stalled problem every block stops there, and the
    # problem behind it is left out in whole; the one ahead of it is done
    sets = [_setup(m, 3, 0), _setup(m, side, 1, npeaks=4, step=1), _setup(m, 4, 2)]
    probs = [s[1] for s in sets]
    probs[0].set_batch_schedule(1, 0)
    assert sets[1][1].nframes > blocks * probs[0].info()["num_sms"]     # more blocks an SM than the kernel can have
    status, outs = _run(sets, 1)
    assert status == [0, 5, 5], status
    _check(sets[0][0], outs[0])
    for (case, p, _), got in zip(sets, mpbp.loss_grad_batched(probs, [s[2] for s in sets])):
        _check(case, got)
        p.sync_status()
