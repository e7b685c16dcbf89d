"""The fused launch over M = 128 problems with scan offsets on some of them: a
block's run then crosses between problems with one probe, with a probe per scan
position and with a probe per frame, reloading them (and prefetching the next
frame's) on either side of the crossing.  Against the FP64 oracle with the
parity tests' tolerances, twice, so that the second call finds what the first
left."""
import numpy as np
import pytest
import torch

import oracle
from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu

# n1, n2, scan side, peaks, per-peak probes, offsets
PROBLEMS = [(140, 150, 9, 2, False, True), (133, 131, 1, 1, False, False), (136, 141, 2, 2, True, True),
            (180, 170, 11, 2, False, False), (129, 128, 1, 2, False, True), (150, 161, 8, 2, True, True)]


def test_runs_across_shifted_probes_match_oracle():
    from paper_2312_14907_gb300 import mpbp
    refs, probs, states = [], [], []
    for i, (n1, n2, side, d, per_peak, shifted) in enumerate(PROBLEMS):
        spec, scan = custom_spec(n1, 128, side, 5, npeaks=d, offset=-4, probe_per_peak=per_peak, n2=n2, seed=40 + i)
        case = Case(spec, scan=scan, state="perturbed", seed=i)
        p = mpbp.Problem.from_spec(spec, scan)
        p.set_probe(torch.from_numpy(case.probe).cuda())
        p.set_data(torch.from_numpy(case.y).cuda())
        if shifted:
            off = np.random.default_rng(i).uniform(-0.5, 0.5, (len(scan), 2))
            p.set_scan_offsets(off)
            o2 = oracle.OracleProblem(spec.n1, spec.n2, spec.ncomp, spec.npeaks, spec.m, scan, spec.G,
                                      spec.phase_scale, probe_per_peak=2)
            refs.append(o2.loss_grad(case.rho, case.u, case.alpha, oracle.frame_probes(o2, case.probe, off), case.y))
        else:
            refs.append(case.oracle_loss_grad())
        probs.append(p)
        states.append(tuple(torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)))
    assert sum(p.nframes for p in probs) > 3 * probs[0].info()["num_sms"]   # runs of three and four frames
    probs[0].set_batch_schedule(1, 0)
    for _ in range(2):
        for (f, gr, gu, ga), p, got in zip(refs, probs, mpbp.loss_grad_batched(probs, states)):
            assert abs(got[0].item() - f) <= 1e-5 * abs(f)
            for a, b in zip(got[1:], (gr, gu, ga)):
                assert rel_l2(a.cpu().numpy(), b) <= 1e-4
            p.sync_status()
