"""The unwrapper's tile and map kernels on whole grids (no mask), where a tile
leaves two to three times the edges of a half-masked one: every map of a size
they serve stays with them (three launches and nothing behind, read off a
captured call), and the result has the bits of the cooperative path (the same
map inside the support of a grid too large for the tiles).  Sizes around the
lists' split between registers and memory and the two cluster sizes; smooth,
noisy, random and constant maps, also side by side in one call; masks that cut
the tiles' rims into as many components as they can; 16 maps."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2312_14907_gb300 import synth

pytestmark = pytest.mark.gpu
BIG = 1024      # 64 x 64 tiles: the cooperative path


def _problem(n1, n2, d):
    from paper_2312_14907_gb300 import mpbp
    g = np.random.default_rng(d).standard_normal((d, 3))
    spec = synth.ProblemSpec("maps", n1, n2, 3, d, 8, 1, 1, g / np.linalg.norm(g, axis=1, keepdims=True),
                             synth.SEED_BASE + 900 + d, bumps=3, straight=1, sigma=1.6, quad=0.04)
    return mpbp.Problem.from_spec(spec, synth.scan_positions(spec))


def _map(kind, n1, n2, rng):
    if kind == "random":
        return rng.uniform(-np.pi, np.pi, (n1, n2)).astype(np.float32)
    if kind == "const":
        return np.full((n1, n2), 0.25, np.float32)
    i, j = np.meshgrid(np.arange(n1), np.arange(n2), indexing="ij")
    p = 0.11 * i + 0.2 * j + 6 * np.sin(i / 23.0)
    if kind == "noisy":
        p = p + 0.9 * rng.standard_normal(p.shape)
    return (np.mod(p + np.pi, 2 * np.pi) - np.pi).astype(np.float32)


def _reference(w, mask):
    """By the cooperative path: inside a larger grid's support, in the same node order."""
    d, n1, n2 = w.shape
    big = _problem(BIG, BIG, d)
    wb, mb = np.zeros((d, BIG, BIG), np.float32), np.zeros((BIG, BIG), np.float32)
    wb[:, 13:13 + n1, 301:301 + n2] = w
    mb[13:13 + n1, 301:301 + n2] = 1.0 if mask is None else mask
    out = big.unwrap_phases(torch.from_numpy(wb).cuda(), torch.from_numpy(mb).cuda())
    big.sync_status()
    return out[:, 13:13 + n1, 301:301 + n2].contiguous()


def _check(w, mask=None):
    p = _problem(w.shape[1], w.shape[2], w.shape[0])
    wd, md = torch.from_numpy(w).cuda(), None if mask is None else torch.from_numpy(mask).cuda()
    got = p.unwrap_phases(wd, md)
    again = p.unwrap_phases(wd, md)
    p.sync_status()
    ref = _reference(w, mask)
    for m in range(w.shape[0]):
        assert torch.equal(got[m], ref[m]), (m, (got[m] - ref[m]).abs().max())
    assert torch.equal(again, got)


# 289 and 306 tiles: the largest of eight and the smallest of sixteen blocks a
# map; 512^2: more edges than sixteen blocks' registers hold; 1,260 tiles
@pytest.mark.parametrize("n1,n2", [(256, 256), (272, 272), (288, 272), (512, 512), (575, 545)])
@pytest.mark.parametrize("kinds", ["smooth", "noisy", "random", "const", "smooth noisy random const"])
def test_whole_grids_agree_with_the_cooperative_path(n1, n2, kinds):
    rng = np.random.default_rng(n1 + n2)
    _check(np.stack([_map(k, n1, n2, rng) for k in kinds.split()]))


def test_sixteen_maps():
    rng = np.random.default_rng(16)
    _check(np.stack([_map(k, 200, 190, rng) for k in ("smooth", "noisy", "random", "const") for _ in range(4)]))


@pytest.mark.parametrize("n1,n2", [(160, 145), (33, 17), (17, 1), (1, 49), (300, 400)])
@pytest.mark.parametrize("cut", ["rims", "rows", "columns"])
def test_most_components_a_tile_can_leave(n1, n2, cut):
    """Pairs of pixels across the tiles' edges on every other line, and lines one pixel wide."""
    rng = np.random.default_rng(n1 * n2)
    i, j = np.meshgrid(np.arange(n1), np.arange(n2), indexing="ij")
    mask = {"rims": (np.isin(j % 16, (0, 15)) & (i % 2 == 0)) | (np.isin(i % 16, (0, 15)) & (j % 2 == 1)),
            "rows": i % 2 == 0, "columns": j % 2 == 0}[cut].astype(np.float32)
    _check(np.stack([_map(k, n1, n2, rng) for k in ("random", "smooth")]), mask)


def _graph_nodes(raw):
    cuda = ctypes.CDLL("libcuda.so.1")
    n = ctypes.c_size_t(0)
    assert cuda.cuGraphGetNodes(ctypes.c_void_p(raw), None, ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("kind", ["smooth", "noisy", "random", "const"])
def test_call_is_three_launches_and_replays(kind):
    rng = np.random.default_rng(3)
    n1, n2 = 300, 280
    p = _problem(n1, n2, 2)
    w = torch.from_numpy(np.stack([_map(kind, n1, n2, rng)] * 2)).cuda()
    out = torch.empty_like(w)
    p.unwrap_phases(w, None, out)               # allocates the workspace
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        p.unwrap_phases(w, None, out)
    assert _graph_nodes(g.raw_cuda_graph()) == 3
    w.copy_(torch.from_numpy(np.stack([_map("noisy", n1, n2, rng), _map("const", n1, n2, rng)])))
    g.instantiate()
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, p.unwrap_phases(w))
    p.sync_status()
