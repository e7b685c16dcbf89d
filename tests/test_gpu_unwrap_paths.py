"""The unwrapper's two paths give the same bits: a map on its own grid (tiles and
one block per map) against the same map inside the support of a grid too large
for that path (one cooperative launch).  Node order, reliabilities and ties are
the same in both, residues or not.  Sizes around the 16 x 16 tiles, several
maps, smooth, noisy and random phases, with and without a mask; and maps that
leave more components than the map kernel can hold."""
import numpy as np
import pytest
import torch

from helpers import custom_spec

pytestmark = pytest.mark.gpu
BIG = 1024      # 64 x 64 tiles: the cooperative path


def _problem(n1, n2, d):
    from paper_2312_14907_gb300 import mpbp
    spec, scan = custom_spec(n1, 8, 1, 1, npeaks=d, offset=0, n2=n2)
    return mpbp.Problem.from_spec(spec, scan)


def _phases(kind, d, n1, n2, rng):
    if kind == "random":
        return rng.uniform(-np.pi, np.pi, (d, n1, n2)).astype(np.float32)
    i, j = np.meshgrid(np.arange(n1), np.arange(n2), indexing="ij")
    p = np.stack([(0.11 + 0.05 * k) * i + (0.2 - 0.03 * k) * j + 6 * np.sin(i / 23.0 + k) for k in range(d)])
    p = p + {"smooth": 0.0, "noisy": 0.9}[kind] * rng.standard_normal(p.shape)
    return (np.mod(p + np.pi, 2 * np.pi) - np.pi).astype(np.float32)


@pytest.mark.parametrize("n1,n2,d", [(1, 1, 1), (3, 50, 2), (15, 17, 1), (16, 16, 3), (33, 31, 2), (64, 80, 16),
                                     (200, 187, 3), (400, 390, 1), (530, 560, 1)])
@pytest.mark.parametrize("kind", ["smooth", "noisy", "random"])
def test_paths_agree(n1, n2, d, kind):
    if d == 16:
        d = 4       # the spec's peaks
    rng = np.random.default_rng(n1 * 1000 + n2)
    w = _phases(kind, d, n1, n2, rng)
    mask = (rng.uniform(size=(n1, n2)) > (0.0 if kind == "smooth" else 0.1)).astype(np.float32)
    mask[: n1 // 3, n2 // 2:] = 0.0
    for m in (None, mask):
        p = _problem(n1, n2, d)
        md = None if m is None else torch.from_numpy(m).cuda()
        got = p.unwrap_phases(torch.from_numpy(w).cuda(), md)
        again = p.unwrap_phases(torch.from_numpy(w).cuda(), md)
        p.sync_status()
        big, o1, o2 = _problem(BIG, BIG, d), 13, 301
        wb = np.zeros((d, BIG, BIG), np.float32)
        mb = np.zeros((BIG, BIG), np.float32)
        wb[:, o1:o1 + n1, o2:o2 + n2] = w
        mb[o1:o1 + n1, o2:o2 + n2] = 1.0 if m is None else m
        ref = big.unwrap_phases(torch.from_numpy(wb).cuda(), torch.from_numpy(mb).cuda())
        big.sync_status()
        ref = ref[:, o1:o1 + n1, o2:o2 + n2]
        assert torch.equal(got, ref), (got - ref).abs().max()
        assert torch.equal(again, got)


def test_too_many_components_fall_back():
    """Isolated pairs of pixels in every third row and column of a grid: components of their own
    that no edge leaves; then a map of 2 x 2 cells of random phase levels, whose lists outgrow shared memory."""
    rng = np.random.default_rng(5)
    n1, n2 = 390, 400
    p = _problem(n1, n2, 1)
    w = rng.uniform(-np.pi, np.pi, (1, n1, n2)).astype(np.float32)
    pairs = np.zeros((n1, n2), np.float32)
    pairs[::3, ::3] = 1.0
    pairs[::3, 1::3] = 1.0
    got = p.unwrap_phases(torch.from_numpy(w).cuda(), torch.from_numpy(pairs).cuda()).cpu().numpy()
    a, b = w[0, ::3, ::3], w[0, ::3, 1::3]
    n = min(a.shape[1], b.shape[1])
    k = np.round((got[0, ::3, 1::3][:, :n] - b[:, :n]) / (2 * np.pi))
    assert np.all(np.abs(got[0, ::3, ::3][:, :n] - a[:, :n]) < 1e-6)
    assert np.all(np.abs(got[0, ::3, 1::3][:, :n] - got[0, ::3, ::3][:, :n]) <= np.pi + 1e-5) and np.abs(k).max() == 1
    # one-pixel-wide zigzag paths: every tile cut into many components
    cells = np.ones((n1, n2), np.float32)
    cells[::2, 1::4] = 0.0
    cells[1::2, 3::4] = 0.0
    got = p.unwrap_phases(torch.from_numpy(w).cuda(), torch.from_numpy(cells).cuda())
    p.sync_status()
    big = _problem(BIG, BIG, 1)
    wb, mb = np.zeros((1, BIG, BIG), np.float32), np.zeros((BIG, BIG), np.float32)
    wb[:, :n1, 32:32 + n2] = w
    mb[:n1, 32:32 + n2] = cells
    ref = big.unwrap_phases(torch.from_numpy(wb).cuda(), torch.from_numpy(mb).cuda())[:, :n1, 32:32 + n2]
    assert torch.equal(got, ref)
