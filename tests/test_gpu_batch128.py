"""The fused launch over M = 128 problems where a block's run of frames crosses
several of them: problems of one frame, of a few and of more than one frame per
SM, with and without a background, shared and per-peak probes, shifted probes,
odd n2.  Each against the FP64 oracle (the parity tests' tolerances), twice, so
that the second call finds what the first left."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu

# n1, n2, scan side, peaks, background, per-peak probes
PROBLEMS = [(140, 150, 9, 3, False, False), (133, 131, 1, 1, True, False), (136, 140, 2, 2, False, True),
            (200, 190, 12, 2, True, True), (129, 128, 1, 2, False, False), (150, 161, 7, 3, True, False)]


@pytest.mark.parametrize("order", [0, 1])
def test_runs_across_problems_match_oracle(order):
    from paper_2312_14907_gb300 import mpbp
    cases, probs, states = [], [], []
    for i, (n1, n2, side, d, bg, per_peak) in enumerate(PROBLEMS):
        spec, scan = custom_spec(n1, 128, side, 5, npeaks=d, offset=-4, probe_per_peak=per_peak, n2=n2, seed=i)
        case = Case(spec, scan=scan, state="perturbed", bg=bg, seed=i)
        p = mpbp.Problem.from_spec(spec, scan)
        p.set_probe(torch.from_numpy(case.probe).cuda())
        p.set_data(torch.from_numpy(case.y).cuda(), None if case.bg is None else torch.from_numpy(case.bg).cuda())
        cases.append(case)
        probs.append(p)
        states.append(tuple(torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)))
    assert sum(p.nframes for p in probs) > 4 * probs[0].info()["num_sms"]   # runs of four and five frames
    probs[0].set_batch_schedule(1, order)
    for _ in range(2):
        outs = mpbp.loss_grad_batched(probs, states)
        for case, p, got in zip(cases, probs, outs):
            f, gr, gu, ga = case.oracle_loss_grad()
            assert abs(got[0].item() - f) <= 1e-5 * abs(f)
            for a, b in zip(got[1:], (gr, gu, ga)):
                assert rel_l2(a.cpu().numpy(), b) <= 1e-4
            p.sync_status()


def test_more_problems_than_a_launch_holds():
    """70 small problems (more than the 48 and 32 of a launch's parameter space) of sides 8 to 128."""
    from paper_2312_14907_gb300 import mpbp
    cases, probs, states = [], [], []
    for i in range(70):
        m = (8, 16, 32, 64, 128)[i % 5] if i % 7 else 32
        spec, scan = custom_spec(m + 5 + i % 3, m, 2, 3, npeaks=1 + i % 4, offset=-1, seed=100 + i)
        case = Case(spec, scan=scan, state="perturbed", seed=i)
        p = mpbp.Problem.from_spec(spec, scan)
        p.set_probe(torch.from_numpy(case.probe).cuda())
        p.set_data(torch.from_numpy(case.y).cuda())
        cases.append(case)
        probs.append(p)
        states.append(tuple(torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)))
    for case, got in zip(cases, mpbp.loss_grad_batched(probs, states)):
        f, gr, gu, ga = case.oracle_loss_grad()
        assert abs(got[0].item() - f) <= 1e-5 * abs(f)
        assert rel_l2(got[1].cpu().numpy(), gr) <= 1e-4 and rel_l2(got[2].cpu().numpy(), gu) <= 1e-4
