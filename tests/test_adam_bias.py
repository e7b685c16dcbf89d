"""Adam's bias corrections for any stored step count: the state is the caller's
device memory, restored from checkpoints as it stands, so a corrupt count may
give a meaningless correction but has to end.  The kernel's own function,
compiled for the host, with exact fractions as the reference; and the same
counts through a step on the GPU."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
B = (0.9, 0.999, 0.0, 0.5)
SMALL = [-300, -6, -2, -1, 0, 1, 2, 3, 200, 1000]
HUGE = [-2 ** 63, -2 ** 62 - 1, -2 ** 40, 2 ** 40, 2 ** 62 + 1, 2 ** 63 - 1]


def _expected(b, t):
    if t > 0:
        return float(1 - Fraction(b) ** t) if t <= 4096 else 1.0   # beyond: b^t below 2^-60 of 1 for b <= 0.999
    if t == 0:
        return 0.0
    if b == 0.0 or t < -4096:
        return -np.inf                                             # 1 / b^|t| beyond FP64
    return float(1 - 1 / Fraction(b) ** -t)


def _check(b, t, got):
    exact = _expected(b, t)
    if np.isinf(exact):
        assert got == exact or got < -1e300, (b, t, got)
    else:
        # an ulp or two of the power, through one division below zero
        assert abs(got - exact) <= 4 * 2.0 ** -52 * max(abs(exact), 1.0 if t < 0 else 0.0), (b, t, got, exact)


def test_every_count_ends(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = tmp_path / "bias.cpp"
    src.write_text('#include <cstdio>\n#include <cstdlib>\n#include "adam_bias.h"\n'
                   "int main(int n, char** v) {\n"
                   "  for (int i = 1; i + 1 < n; i += 2)\n"
                   '    std::printf("%.17g\\n", mpbp::one_minus_pow(std::atof(v[i]), std::atoll(v[i + 1])));\n}\n')
    exe = str(tmp_path / "bias")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2312_14907_gb300", "csrc"), "-o", exe, str(src)], check=True)
    calls = [(b, t) for b in B for t in SMALL + HUGE]
    args = [s for b, t in calls for s in (repr(b), str(t))]
    out = subprocess.run([exe] + args, capture_output=True, text=True, check=True, timeout=20).stdout.split()
    assert len(out) == len(calls)
    for (b, t), got in zip(calls, out):
        _check(b, t, float(got))


@pytest.mark.gpu
@pytest.mark.parametrize("t", [-2 ** 63, -300, -2, -1, 0, 2 ** 63 - 1])
def test_stored_count_of_any_value(t):
    import torch
    from helpers import Case, custom_spec
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(21, 8, 3, 4, npeaks=2, offset=0)
    case = Case(spec, scan=scan, state="perturbed")
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    x = [torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)]
    st = p.adam_init(beta1=0.9, beta2=0.999)
    h = p.read_adam_state(st)
    h.t = t
    st.copy_(torch.frombuffer(bytearray(h), dtype=torch.uint8))
    p.adam_step(None, torch.zeros_like(x[0]), x[1].clone(), torch.zeros_like(x[2]), st)
    h = p.read_adam_state(st)
    nxt = t + 1 if t < 2 ** 63 - 1 else -2 ** 63
    assert h.t == nxt
    _check(0.9, nxt, h.bc1)
    _check(0.999, nxt, h.bc2)
