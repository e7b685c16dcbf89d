"""Batched calls whose problems share output buffers: the assembly then runs
problem by problem, so that the losses are every problem's own and a shared
buffer holds the last one's result, as with one call after the other."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shared", ["rho", "u", "alpha", "all", "overlap", "input"])
@pytest.mark.parametrize("m", [32, 128])
def test_shared_outputs_hold_the_last_problems(m, shared):
    from paper_2312_14907_gb300 import mpbp
    cases, probs, states = [], [], []
    for i in range(4):
        spec, scan = custom_spec(300, m, 3, m // 2, npeaks=3, offset=0, seed=i)
        case = Case(spec, scan=scan, state="perturbed", seed=i)
        p = mpbp.Problem.from_spec(spec, scan)
        p.set_probe(torch.from_numpy(case.probe).cuda())
        p.set_data(torch.from_numpy(case.y).cuda())
        cases.append(case)
        probs.append(p)
        states.append(tuple(torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)))
    n1 = n2 = 300
    new = lambda: [torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty((n1, n2), device="cuda"),
                   torch.empty((3, n1, n2), device="cuda"), torch.empty(3, dtype=torch.float64, device="cuda")]
    outs = [new() for _ in probs]
    which = {"rho": (1,), "u": (2,), "alpha": (3,), "all": (1, 2, 3)}.get(shared, ())
    for o in outs[:-1]:
        for q in which:
            o[q] = outs[-1][q]
    if shared == "overlap":      # problem 3's df/drho over the end of problem 0's and the start of problem 1's
        pool = torch.empty((3 * n1, n2), device="cuda")
        outs[0][1], outs[1][1], outs[3][1] = pool[:n1], pool[n1:2 * n1], pool[n1 // 2:n1 // 2 + n1]
    if shared == "input":        # problem 3's df/drho over problem 0's density, read before it
        outs[3][1] = states[0][0]
    for _ in range(3):
        if shared == "input":
            states[0][0].copy_(torch.from_numpy(cases[0].rho))
        mpbp.loss_grad_batched(probs, states, [tuple(o) for o in outs])
        for i, (case, o) in enumerate(zip(cases, outs)):
            f, gr, gu, ga = case.oracle_loss_grad()
            assert abs(o[0].item() - f) <= 1e-5 * abs(f)
            last = i == len(cases) - 1
            if last or 1 not in which:
                if shared == "overlap" and i < 2:
                    keep = slice(0, n1 // 2) if i == 0 else slice(n1 // 2, n1)
                    assert rel_l2(o[1].cpu().numpy()[keep], gr[keep]) <= 1e-4
                else:
                    assert rel_l2(o[1].cpu().numpy(), gr) <= 1e-4
            if last or 2 not in which:
                assert rel_l2(o[2].cpu().numpy(), gu) <= 1e-4
            if last or 3 not in which:
                assert rel_l2(o[3].cpu().numpy(), ga) <= 1e-4
    for p in probs:
        p.sync_status()
