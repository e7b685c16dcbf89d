"""Objects with an odd number of columns, whose workspace rows are padded by
one value: every kernel that reads them against the FP64 oracle (tolerances as
the parity tests': loss 1e-5, gradients and objects 1e-4 / 1e-5)."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu


def _setup(m, n2, npeaks=2, seed=0):
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(2 * m + 3, m, 4, m // 3 + 1, npeaks=npeaks, offset=-3, n2=n2, seed=seed)
    case = Case(spec, scan=scan, state="perturbed", seed=seed)
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    return case, p, [torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)]


def _check(case, got, frames=None):
    f, gr, gu, ga = case.oracle_loss_grad(frames=frames)
    assert abs(got[0].item() - f) <= 1e-5 * abs(f)
    assert rel_l2(got[1].cpu().numpy(), gr) <= 1e-4
    assert rel_l2(got[2].cpu().numpy(), gu) <= 1e-4
    assert rel_l2(got[3].cpu().numpy(), ga) <= 1e-4


@pytest.mark.parametrize("m", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("wide", [1, 0])
def test_odd_columns_match_oracle(m, wide):
    from paper_2312_14907_gb300 import mpbp
    case, p, x = _setup(m, 2 * m + 5 if wide else m + 1)   # the second: narrower than a tile
    _check(case, p.loss_grad(*x))
    frames = np.array([5, 0, 31, 5, 17], np.int32)
    _check(case, p.loss_grad(*x, frames=torch.from_numpy(frames).cuda()), frames)
    f = case.oracle_loss_grad()[0]
    assert abs(p.loss(*x).item() - f) <= 1e-5 * abs(f)
    assert rel_l2(p.forward(*x).cpu().numpy(), case.oracle.forward(case.rho, case.u, case.alpha, case.probe)) <= 1e-5
    O = p.object_build(*x).cpu().numpy()      # the caller's buffer has no padding
    assert rel_l2(O, case.oracle.object_build(case.rho, case.u, case.alpha)) <= 1e-5
    if m >= 32:
        p.set_precision(mpbp.PRECISION_TC_SPLIT16)
        _check(case, p.loss_grad(*x))
    p.sync_status()


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_batch_with_odd_columns_matches_oracle(mode):
    from paper_2312_14907_gb300 import mpbp
    sets = [_setup(m, n2, npeaks=3, seed=i)
            for i, (m, n2) in enumerate([(32, 71), (64, 133), (128, 261), (32, 64), (64, 130), (128, 258)])]
    probs = [s[1] for s in sets]
    probs[0].set_batch_schedule(mode, 0)
    outs = mpbp.loss_grad_batched(probs, [tuple(s[2]) for s in sets])
    for (case, p, _), got in zip(sets, outs):
        _check(case, got)
        p.sync_status()
