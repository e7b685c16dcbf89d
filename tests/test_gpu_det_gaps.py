"""The deterministic gradient where a strip's frames leave rows between them that
none reaches (its pieces are then cleared on every call), where they just touch,
and where pieces lie beside, across and off the grid's edges: against the FP64
oracle (the parity tests' tolerances) and bit for bit on repetition, on a grid
whose sides are no multiples of the 8 x 32 pixels a block sums."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [64, 128])
@pytest.mark.parametrize("jump", [-1, 0, 1, 37])     # rows between two frames of a strip, beyond touching
def test_gaps_match_oracle(m, jump):
    from paper_2312_14907_gb300 import mpbp
    n1, n2 = 3 * m + 45, m + 77 + (m + 77) % 2
    rows = [-m // 2, -m // 2 + m + jump, -m // 2 + 2 * (m + jump), -m // 2 + 3 * (m + jump)]
    cols = [-m // 3, 5, 30, n2 - m // 2]
    scan = np.array([[r, c] for c in cols for r in rows] + [[2 * m, -m - 3], [n1 + 5, 3], [-m, 2]], np.int32)
    scan = np.concatenate([scan] * 12)      # repeats: several frames of a block share a strip
    spec, _ = custom_spec(n1, m, 1, 1, npeaks=2, n2=n2)
    case = Case(spec, scan=scan, state="perturbed")
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    p.set_schedule(1)
    p.set_deterministic(True)
    x = [torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)]
    first = [t.clone() for t in p.loss_grad(*x)]
    f, gr, gu, ga = case.oracle_loss_grad()
    assert abs(first[0].item() - f) <= 1e-5 * abs(f)
    for a, b in zip(first[1:], (gr, gu, ga)):
        assert rel_l2(a.cpu().numpy(), b) <= 1e-4
    y = [t * 1.5 for t in x]
    p.loss_grad(*y)                          # other values in the pieces
    for a, b in zip(first, p.loss_grad(*x)):
        assert torch.equal(a.view(torch.uint8), b.view(torch.uint8))
    p.sync_status()
