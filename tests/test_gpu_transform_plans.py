"""Plane-transform plans: every kind of N' (radices, stages, threads per row) against the exact DFT.

N' runs over first radices 8 .. 28, middle radices 6 .. 21, two to four stages, one and
several TMA boxes per row, and the compile-time sizes; shared rows (several CTAs per image
row) are compared with unshared sums of the same planes.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import REL_TOL, rel, tol_for
from oracle.geometry import make_geometry
from paper_2101_11172_gb300 import synth

pytestmark = pytest.mark.gpu

# (N, x0, N'): two stages, then three (448 = 28 16 inverse, 8 8 7 forward), four and the largest
SIZES = [(16, 0.25, 32), (48, 0.25, 96), (80, 0.25, 160), (144, 0.25, 288), (200, 0.25, 448), (240, 0.25, 480),
         (256, 0.25, 512), (288, 0.25, 576), (336, 0.25, 672), (400, 0.25, 800), (512, 0.25, 1024), (784, 0.25, 1568),
         (864, 0.25, 1728), (1000, 0.25, 2016), (1024, 0.25, 2048), (1296, 0.25, 2592), (1680, 0.25, 3360),
         (2048, 0.25, 4096), (2160, 0.25, 4320), (3024, 0.25, 6048), (4096, 0.375, 5600)]


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _case(N, fov, M, w_half, seed):
    rng = synth.rng_for(0, 7000 + seed)
    uvw = synth.disc_uvw(M, 0.45 * N / fov, w_half, rng)
    return uvw, rng


@pytest.mark.parametrize("N,x0,Np", SIZES)
def test_plan_against_dft(dev, N, x0, Np):
    from paper_2101_11172_gb300.wstack import Plan
    W, fov, M = 7, 0.2, 400
    # about ten planes: n_scale w spans a few planes
    w_half = 2.0 * (2 * x0) / (2 * (fov / 2) ** 2) * 2
    uvw, rng = _case(N, fov, M, w_half, Np)
    w_min, w_max = float(uvw[:, 2].min()), float(uvw[:, 2].max())
    g = make_geometry(N, x0, W, fov, w_min, w_max)
    assert g.Np == Np
    # sources and sampled pixels over the whole image, its corners and centre included
    edge = np.array([0, N // 2, N - 1, (N - 1) * N, N * N - 1, (N // 2) * N + N // 2])
    pix = np.unique(np.concatenate([edge, rng.choice(N * N, size=min(120, N * N // 2), replace=False)]))
    image = np.zeros(N * N, dtype=np.complex128)
    image[pix] = synth.complex_normal(pix.size, rng)
    vis = synth.complex_normal(M, rng)
    l = (pix % N - N // 2) * (fov / N)
    m = (pix // N - N // 2) * (fov / N)
    lmn = np.stack([l, m, -(l * l + m * m) / (1 + np.sqrt(1 - l * l - m * m))], 1)
    phase = 2 * np.pi * (uvw @ lmn.T)
    v_ref = np.exp(-1j * phase) @ image[pix]
    d_ref = np.exp(1j * phase).T @ vis
    tol = tol_for(W, g.x0)
    with Plan(N, x0, W, fov, w_min, w_max, device=dev) as p:
        assert p.Np == Np
        t_uvw = torch.from_numpy(uvw).to(dev)
        v = p.degrid(torch.from_numpy(image.reshape(N, N)).to(torch.complex64).to(dev), t_uvw).cpu().numpy()
        d = p.grid(t_uvw, torch.from_numpy(vis).to(torch.complex64).to(dev)).cpu().numpy().ravel()[pix]
    print(Np, rel(v, v_ref), rel(d, d_ref), tol)
    assert rel(v, v_ref) < tol
    assert rel(d, d_ref) < tol


@pytest.mark.parametrize("N,chunk", [(64, 0), (64, 16), (256, 0), (256, 24), (200, 0)])
def test_shared_rows(dev, monkeypatch, N, chunk):
    """Rows shared by several CTAs give the sum over all planes, in one chunk or several."""
    from paper_2101_11172_gb300.wstack import Plan
    W, fov, M = 7, 0.2, 2000
    uvw, rng = _case(N, fov, M, 1500.0, N + chunk)
    w_min, w_max = float(uvw[:, 2].min()), float(uvw[:, 2].max())
    vis = synth.complex_normal(M, rng)
    pix = rng.choice(N * N, size=300, replace=False)
    l, m = (pix % N - N // 2) * (fov / N), (pix // N - N // 2) * (fov / N)
    lmn = np.stack([l, m, -(l * l + m * m) / (1 + np.sqrt(1 - l * l - m * m))], 1)
    d_ref = np.exp(2j * np.pi * (uvw @ lmn.T)).T @ vis
    if chunk:
        monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(chunk))
    with Plan(N, 0.25, W, fov, w_min, w_max, device=dev) as p:
        assert p.Nw > 60 and (p.planes_per_chunk == chunk or not chunk)
        t_uvw, t_vis = torch.from_numpy(uvw).to(dev), torch.from_numpy(vis).to(torch.complex64).to(dev)
        for _ in range(2):                        # the row counters are zero again after a call
            d = p.grid(t_uvw, t_vis).cpu().numpy().ravel()[pix]
            assert rel(d, d_ref) < REL_TOL
