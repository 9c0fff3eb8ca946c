"""Tensor-core gridding: every width it serves, at the sizes where its tiling and staging have edges.

Against the FP64 oracle's Algorithm 5: bins of 1 to more than 64 entries (the staged chunk), few and
many planes, plane chunks that cut a column, tile columns on the wrapped edges of the grid, N' = 32
(two tiles, every footprint near an edge), real-sky folding, and the tile rows that keep the other kernel.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import assert_elementwise, case, oracle_pair, rel, tol_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _grid(c, dev, flags=0):
    from paper_2101_11172_gb300.wstack import Plan
    with Plan(c["N"], c["x0"], c["W"], c["fov"], c["w_min"], c["w_max"], flags=flags, device=dev) as p:
        return p.grid(torch.from_numpy(c["uvw"]).to(dev),
                      torch.from_numpy(c["vis"]).to(torch.complex64).to(dev)).cpu().numpy()


@pytest.mark.parametrize("W", range(1, 10))
@pytest.mark.parametrize("N,M,wfac", [(16, 700, 4.0), (64, 1, 0.0), (64, 5, 8.0), (64, 3000, 30.0), (96, 40_000, 3.0)])
def test_widths_and_bins(dev, W, N, M, wfac):
    c = case(N=N, M=M, W=W, wfac=wfac, seed=100 * W + N)
    g, _, _, d_ref = oracle_pair(c)
    tol = tol_for(W, g.x0)
    d = _grid(c, dev)
    assert rel(d, d_ref) < tol
    assert_elementwise(d, d_ref, tol, f"W={W} N={N} M={M}")


@pytest.mark.parametrize("W,chunk", [(7, 8), (7, 24), (9, 8), (4, 16)])
def test_plane_chunks(dev, monkeypatch, W, chunk):
    """Planes in chunks: bins before a chunk reach into it, and tiles outside it are not written."""
    c = case(N=64, M=4000, W=W, wfac=40.0, seed=W + chunk)
    g, _, _, d_ref = oracle_pair(c)
    monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(chunk))
    assert rel(_grid(c, dev), d_ref) < tol_for(W, g.x0)


def test_one_crowded_cell_and_edges(dev):
    """Many visibilities in one bin (chunks of 64), and footprints across every edge of the grid."""
    c = case(N=64, M=3000, W=7, wfac=10.0, seed=77)
    scale = (0.5 * c["N"] / c["fov"]) / 1.0
    c["uvw"][:1500, :2] = c["uvw"][0, :2] * 0.3 + 1e-3 * c["uvw"][:1500, :2]
    c["uvw"][:1500, 2] = c["uvw"][0, 2]
    rng = np.random.default_rng(5)
    edge = rng.choice([-1.0, 0.0, 1.0], size=(1500, 2)) * scale * 2 + rng.uniform(-4, 4, (1500, 2)) / c["fov"] / 4
    c["uvw"][1500:, :2] = edge
    g, _, _, d_ref = oracle_pair(c)
    d = _grid(c, dev)
    assert rel(d, d_ref) < tol_for(7, g.x0)
