"""The Adam moments saved into arrays that share memory (a caller after some of
them may pass one scratch array for the rest): each array holds its moments
where no later one overlaps it, the later one where it does; and saved and
loaded moments are the same bits at lengths that leave every remainder."""
import numpy as np
import pytest
import torch

from helpers import Case, custom_spec

pytestmark = pytest.mark.gpu


def _stepped(n1, n2, npeaks, ncomp=3):
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(n1, 8, 3, 4, npeaks=npeaks, ncomp=ncomp, offset=0, n2=n2)
    case = Case(spec, scan=scan, state="perturbed")
    p = mpbp.Problem.from_spec(spec, scan)
    p.set_probe(torch.from_numpy(case.probe).cuda())
    p.set_data(torch.from_numpy(case.y).cuda())
    st = p.adam_init()
    v = [torch.from_numpy(np.log(np.maximum(case.rho, 0.1))).cuda(), torch.from_numpy(case.u).cuda(),
         torch.zeros(npeaks, device="cuda")]
    p.adam_step(None, *v, st)
    p.sync_status()
    return p


def _raw_get(p, out):
    from paper_2312_14907_gb300 import mpbp
    lib = mpbp.load()
    s = lib.mpbp_adam_get_state(p._h, *[t.data_ptr() for t in out], mpbp._stream())
    assert s == 0
    torch.cuda.synchronize()


def test_shared_targets():
    p = _stepped(1024, 1024, 3)
    ref = p.adam_get_state()
    n = 1024 * 1024
    scratch = torch.empty(3 * n, device="cuda")
    # m_chi and v_chi into the front of the scratch, m_u over both, v_u over m_u; m_alpha and v_alpha shared
    a = torch.empty(3, dtype=torch.float64, device="cuda")
    for _ in range(5):
        scratch.fill_(-1.0)
        _raw_get(p, (scratch[:n], scratch[n:2 * n], scratch, scratch, a, a))
        assert torch.equal(scratch, ref[3].reshape(-1)) and torch.equal(a, ref[5])
        # v_chi over the second half of m_chi
        scratch.fill_(-1.0)
        out = [torch.empty_like(t) for t in ref]
        _raw_get(p, (scratch[:n], scratch[n // 2:n // 2 + n], *out[2:]))
        assert torch.equal(scratch[:n // 2], ref[0].reshape(-1)[:n // 2])
        assert torch.equal(scratch[n // 2:n // 2 + n], ref[1].reshape(-1))
        for x, y in zip(out[2:], ref[2:]):
            assert torch.equal(x, y)


@pytest.mark.parametrize("n1,n2,npeaks", [(9, 9, 1), (9, 10, 2), (11, 13, 3), (40, 33, 4)])
def test_saved_and_loaded_moments_are_the_same_bits(n1, n2, npeaks):
    p = _stepped(n1, n2, npeaks)
    ref = p.adam_get_state()
    rng = torch.Generator(device="cuda").manual_seed(n1)
    put = [torch.rand(t.shape, dtype=t.dtype, device="cuda", generator=rng) for t in ref]
    p.adam_set_state(put)
    # targets off a 16-byte boundary as well
    for off in (0, 1):
        got = []
        for t in ref:
            buf = torch.empty(t.numel() + 4, dtype=t.dtype, device="cuda")
            got.append(buf[off:off + t.numel()])
        _raw_get(p, got)
        for x, y in zip(got, put):
            assert torch.equal(x, y.reshape(-1))
    p.sync_status()
