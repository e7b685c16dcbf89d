"""The kernels' two ways of taking their inputs, each forced and each named by
the context: TMA tile and bulk copies (even n2; odd n2 over padded rows) and
per-element cp.async, through every entry point that has both.  Against the
FP64 oracle at the parity tests' tolerances (loss 1e-5, gradients 1e-4,
intensities 1e-5)."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec, rel_l2

pytestmark = pytest.mark.gpu


def _setup(spec, scan, element, seed=0, **kw):
    from paper_2312_14907_gb300 import mpbp
    case = Case(spec, scan=scan, state="perturbed", seed=seed, **kw)
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda(), None if case.bg is None else torch.from_numpy(case.bg).cuda())
    if element:
        p.set_test_element_copies()
    want = mpbp.COPIES_ELEMENT if element else (mpbp.COPIES_TILE_PADDED if spec.n2 % 2 else mpbp.COPIES_TILE)
    assert p.input_copies() == (want, want)
    return case, p, [torch.from_numpy(a).cuda() for a in (case.rho, case.u, case.alpha)]


def _check(case, got, frames=None):
    f, gr, gu, ga = case.oracle_loss_grad(frames=frames)
    assert abs(got[0].item() - f) <= 1e-5 * abs(f)
    for a, b in zip(got[1:], (gr, gu, ga)):
        assert rel_l2(a.cpu().numpy(), b) <= 1e-4


def _all_entries(case, p, x, host):
    _check(case, p.loss_grad(*x))
    frames = np.random.default_rng(1).permutation(p.nframes)[: max(1, 2 * p.nframes // 3)].astype(np.int32)
    fd = torch.from_numpy(frames).cuda()
    _check(case, p.loss_grad(*x, frames=fd), frames)
    for fr, fdev in ((None, None), (frames, fd)):
        f = case.oracle_loss_grad(frames=fr)[0]
        assert abs(p.loss(*x, frames=fdev).item() - f) <= 1e-5 * abs(f)
    I = p.forward(*x).cpu().numpy()
    I_ref = case.oracle.forward(case.rho, case.u, case.alpha, case.probe, bg=case.bg)
    d = np.linalg.norm((I - I_ref).reshape(p.nframes, -1), axis=1)
    assert np.all(d <= 1e-5 * np.linalg.norm(I_ref.reshape(p.nframes, -1), axis=1))
    if host:
        h = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory()
        for y in (case.y, case.y.astype(np.uint16)):
            _check(case, p.loss_grad_host(h(case.rho), h(case.u), h(case.alpha), y=h(y)))
    p.sync_status()


@pytest.mark.parametrize("element", [False, True])
@pytest.mark.parametrize("odd", [0, 1])
@pytest.mark.parametrize("m,schedule", [(32, 1), (64, 1), (128, 0), (128, 1)])
def test_every_entry_point(m, schedule, odd, element):
    spec, scan = custom_spec(2 * m + 6, m, 3, m // 2 + 1, npeaks=2, offset=-3, n2=2 * m + 8 - odd)
    for bg in (False, True):
        case, p, x = _setup(spec, scan, element, bg=bg)
        p.set_fft_schedule(schedule)
        _all_entries(case, p, x, host=not bg)


# more frames than two a block (608 blocks at M = 64, 152 at M = 128), so that
# a block reuses its buffers, and the copies' barrier its phases
@pytest.mark.parametrize("element", [False, True])
@pytest.mark.parametrize("m,schedule,n1,n2,side,step", [(64, 1, 170, 199, 26, 5), (128, 0, 256, 255, 13, 10),
                                                        (128, 1, 256, 255, 13, 10), (128, 1, 256, 256, 13, 10)])
def test_steady_state(m, schedule, n1, n2, side, step, element):
    spec, scan = custom_spec(n1, m, side, step, npeaks=2, offset=-6, n2=n2)
    case, p, x = _setup(spec, scan, element)
    p.set_fft_schedule(schedule)
    assert spec.nframes > 2 * p.info()["frames_grid"]
    _all_entries(case, p, x, host=False)


@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_batch(mode):
    from paper_2312_14907_gb300 import mpbp
    sets = []
    for i, (m, n2) in enumerate([(32, 71), (64, 133), (128, 261), (32, 64), (64, 130), (128, 258)]):
        spec, scan = custom_spec(2 * m + 3, m, 4, m // 3 + 1, npeaks=3, offset=-3, n2=n2, seed=i)
        sets.append(_setup(spec, scan, element=i != 3, seed=i))     # one of side 32 with tile copies among them
    probs = [s[1] for s in sets]
    probs[0].set_batch_schedule(mode, 0)
    for switch in (None, False, True):      # a plan follows a change of the copies
        if switch is not None:
            for p in probs:
                p.set_test_element_copies(switch)
        for (case, p, _), got in zip(sets, mpbp.loss_grad_batched(probs, [tuple(s[2]) for s in sets])):
            _check(case, got)
            p.sync_status()


def test_switch_and_deterministic_mode():
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(136, 64, 3, 33, npeaks=2, offset=-3)
    case, p, x = _setup(spec, scan, True)
    with pytest.raises(mpbp.MPBPError):
        p.set_deterministic(True)
    p.set_test_element_copies(False)
    assert p.input_copies() == (mpbp.COPIES_TILE,) * 2
    p.set_deterministic(True)
    with pytest.raises(mpbp.MPBPError):
        p.set_test_element_copies(True)
    assert p.input_copies() == (mpbp.COPIES_TILE,) * 2
    _check(case, p.loss_grad(*x))
    p.sync_status()
    small, s2 = custom_spec(40, 16, 3, 6, npeaks=2, offset=0)
    q = mpbp.Problem.from_spec(small, s2)
    assert q.input_copies() == (mpbp.COPIES_ELEMENT,) * 2      # M <= 16 has no tile copies
