"""The gradient assembly with 4, 8 or 16 peaks held in registers, in each of
its forms, against the FP64 oracle (the parity tests' tolerances), and the
bias corrections of the Adam step against exact powers."""
import ctypes
from fractions import Fraction

import numpy as np
import pytest
import torch

from helpers import Case, rel_l2
from paper_2312_14907_gb300 import synth

pytestmark = pytest.mark.gpu


def _case(d):
    g = np.random.default_rng(d).standard_normal((d, 3))
    spec = synth.ProblemSpec("peaks", 21, 19, 3, d, 8, 4, 3, g / np.linalg.norm(g, axis=1, keepdims=True),
                             synth.SEED_BASE + 700 + d, bumps=3, straight=1, sigma=1.6, quad=0.04)
    from paper_2312_14907_gb300 import mpbp
    case = Case(spec, state="perturbed")
    p = mpbp.Problem.from_spec(spec, case.scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    return case, p, [torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)]


@pytest.mark.parametrize("d", [1, 4, 5, 8, 9, 16])
def test_peak_counts_match_oracle(d):
    case, p, x = _case(d)
    f, gr, gu, ga = case.oracle_loss_grad()
    got = p.loss_grad(*x)
    assert abs(got[0].item() - f) <= 1e-5 * abs(f)
    for a, b in zip(got[1:], (gr, gu, ga)):
        assert rel_l2(a.cpu().numpy(), b) <= 1e-4
    # the phase form at the phases u defines: df/du is their chain rule
    ps = case.spec.phase_scale
    phi = torch.einsum("mc,cij->mij", torch.from_numpy(case.spec.G * ps).cuda(), x[1].double()).float().contiguous()
    fp, grp, gphi, gap = p.loss_grad_phases(x[0], phi, x[2])
    assert abs(fp.item() - f) <= 1e-5 * abs(f)
    assert rel_l2(grp.cpu().numpy(), gr) <= 1e-4
    back = np.einsum("mc,mij->cij", case.spec.G * ps, gphi.cpu().numpy().astype(np.float64))
    assert rel_l2(back, gu) <= 1e-4
    # one step of gradient descent from the start: x - t w g
    t0, w = 1e-3 / abs(gr).max(), {"w_rho": 1.0, "w_u": 0.05, "w_alpha": 0.01}
    st = p.step_init(t0, **w)
    y = [t.clone() for t in x]
    p.step(*y, st)
    assert rel_l2((y[0] - x[0]).cpu().numpy(), -t0 * gr) <= 1e-3     # differences of FP32 values near 1
    s = p.read_state(st)
    assert abs(s.f_last - f) <= 1e-5 * abs(f) and s.accepted == 1
    # one Adam step from zero moments: m = (1 - beta1) g, v = (1 - beta2) g^2
    at = torch.log(x[2].clamp(min=1e-2)).contiguous()
    chi = torch.log(x[0].clamp(min=0.1)).contiguous()
    alpha = np.exp(at.cpu().numpy().astype(np.float64))
    alpha[0] = 1.0
    rho = np.exp(chi.cpu().numpy().astype(np.float64))
    fo, go, guo, gao = case.oracle_loss_grad(rho=rho, alpha=alpha)
    ast = p.adam_init()
    v = [chi.clone(), x[1].clone(), at.clone()]
    p.adam_step(None, *v, ast)
    m_chi, v_chi, m_u, v_u, m_a, v_a = [t.cpu().numpy().astype(np.float64) for t in p.adam_get_state()]
    assert rel_l2(m_chi, 0.1 * rho * go) <= 1e-4 and rel_l2(m_u, 0.1 * guo) <= 1e-4
    assert rel_l2(v_chi, 1e-3 * (rho * go) ** 2) <= 3e-4 and rel_l2(v_u, 1e-3 * guo ** 2) <= 3e-4
    if d > 1:
        assert rel_l2(m_a[1:], 0.1 * (alpha * gao)[1:]) <= 1e-4
    assert v[2][0] == at[0]
    p.sync_status()


@pytest.mark.parametrize("t", [1, 2, 3, 200, 4095, 10**6, 2**40])
def test_bias_corrections(t):
    case, p, x = _case(4)
    b1, b2 = 0.9, 0.999
    st = p.adam_init(beta1=b1, beta2=b2)
    h = p.read_adam_state(st)
    h.t = t - 1
    st.copy_(torch.frombuffer(bytearray(h), dtype=torch.uint8))
    p.adam_step(None, torch.zeros_like(x[0]), x[1].clone(), torch.zeros_like(x[2]), st)
    h = p.read_adam_state(st)
    assert h.t == t
    for b, got in ((b1, h.bc1), (b2, h.bc2)):
        exact = float(1 - Fraction(b) ** t) if t <= 4095 else 1.0      # 0.999^10^6 < 1e-400
        assert abs(got - exact) <= 4 * 2.0 ** -52 * exact              # an ulp or two of the result
