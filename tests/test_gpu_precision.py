"""FP32 rounding of single stages, where a whole call's error bar would not show it."""
import numpy as np
import pytest
import torch

from gpu_helpers import rel
from paper_2101_11172_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


# N' = 5120 and 4096 where the row kernel keeps no stepped screen
@pytest.mark.parametrize("N,x0", [(2560, 0.25), (3072, 0.375)])
def test_large_rows_screen_every_plane_exactly(dev, monkeypatch, N, x0):
    """Each plane's screen is a function of the plane alone: visibilities whose footprint lies within one
    chunk come out bit for bit the same however the planes are dealt out.  (A screen stepped from plane to
    plane rounds by its distance from the last exact one.)"""
    from paper_2101_11172_gb300.wstack import Plan
    W, fov, M, w_half = 4, 0.3, 4000, 400.0
    rng = synth.rng_for(0, 9100)
    uvw = synth.disc_uvw(M, 0.45 * N / fov, w_half, rng)
    image = torch.from_numpy(synth.complex_normal(N * N, rng).reshape(N, N)).to(torch.complex64).to(dev)
    t_uvw = torch.from_numpy(uvw).to(dev)
    out = []
    for chunk in (0, 24):
        if chunk:
            monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(chunk))
        with Plan(N, x0, W, fov, -w_half, w_half, device=dev) as p:
            assert p.Nw > 24 and (p.planes_per_chunk == chunk or not chunk)
            out.append(p.degrid(image, t_uvw).cpu().numpy())
            first = np.floor(uvw[:, 2] * p.nscale + 0.5 * W) - (W - 1) - p.t_lo
    whole = first % 24 <= 24 - W
    assert 0.5 < whole.mean() < 1.0
    assert np.array_equal(out[0][whole], out[1][whole])


def _grid(p, uvw, vis):
    return p.grid(uvw, vis.to(p.cdtype)).to(torch.complex128).cpu().numpy()


@pytest.mark.parametrize("N,W,M", [(64, 7, 1000), (256, 7, 10), (256, 7, 1000), (256, 8, 10_000), (256, 4, 1000),
                                   (128, 9, 3000)])
def test_gridding_products_are_fp32(dev, N, W, M):
    """Against an FP64 plan, the default mode is no further off than the deterministic one, whose contributions
    are FP32 products (three roundings each) summed exactly: here one rounding fewer a product and a sum or two
    per cell, so 5 % is left for the sums."""
    from paper_2101_11172_gb300 import WS_FLAG_DETERMINISTIC, WS_FLAG_FP64
    from paper_2101_11172_gb300.wstack import Plan
    sq = np.zeros(2)
    for seed in range(4):
        rng = synth.rng_for(0, 9200 + 10 * W + seed)
        uvw = torch.from_numpy(synth.disc_uvw(M, 0.45 * N / 0.2, 1.0, rng)).to(dev)
        vis = torch.from_numpy(synth.complex_normal(M, rng).astype(np.complex64).astype(np.complex128)).to(dev)
        d = []
        for flags in (WS_FLAG_FP64, 0, WS_FLAG_DETERMINISTIC):
            with Plan(N, 0.25, W, 0.2, -1.0, 1.0, flags=flags, device=dev) as p:
                d.append(_grid(p, uvw, vis))
        sq += rel(d[1], d[0]) ** 2, rel(d[2], d[0]) ** 2
    print(N, W, M, np.sqrt(sq / 4))
    assert sq[0] <= 1.05 ** 2 * sq[1]


@pytest.mark.parametrize("power", [-110, 90])
def test_gridding_keeps_its_digits_at_every_scale(dev, power):
    """Visibilities scaled by a power of two give the image scaled by it, up to the order of the sums
    (about 1e-7): only contributions below 2^-126, 2^-16 of these visibilities, lose digits."""
    from paper_2101_11172_gb300.wstack import Plan
    N, W, M = 256, 7, 5000
    rng = synth.rng_for(0, 9300)
    uvw = torch.from_numpy(synth.disc_uvw(M, 0.45 * N / 0.2, 1.0, rng)).to(dev)
    vis = torch.from_numpy(synth.complex_normal(M, rng).astype(np.complex64).astype(np.complex128)).to(dev)
    with Plan(N, 0.25, W, 0.2, -1.0, 1.0, device=dev) as p:
        one, scaled = _grid(p, uvw, vis), _grid(p, uvw, vis * 2.0 ** power)
    assert rel(scaled * 2.0 ** -power, one) < 1.4e-7


@pytest.mark.parametrize("N,Np", [(768, 1536), (1296, 2592), (1536, 3072), (2160, 4320), (2592, 5184)])
def test_inverse_plans_are_as_accurate_as_the_forward_ones(dev, N, Np):
    """Larger radices in the inverse plans, with stages of 6, 12 and 16 where the forward ones have 3s and 8s, cost
    no accuracy: gridding is as far from the exact DFT as degridding on the same plan (5 % for the sampling; the
    same transform in both directions gives ratios of 0.94 to 1.02 at these sizes)."""
    from paper_2101_11172_gb300.wstack import Plan
    W, fov, M, n_pix = 8, 0.3, 20_000, 3000
    err = np.zeros(2)
    with Plan(N, 0.25, W, fov, -100.0, 100.0, device=dev) as p:
        assert p.Np == Np
        for seed in range(4):
            rng = synth.rng_for(0, 9400 + Np + seed)
            uvw = torch.from_numpy(synth.disc_uvw(M, 0.45 * N / fov, 100.0, rng)).to(dev)
            vis = torch.from_numpy(synth.complex_normal(M, rng).astype(np.complex64)).to(dev)
            pix = torch.from_numpy(rng.choice(N * N, size=n_pix, replace=False)).to(dev)
            amp = torch.from_numpy(synth.complex_normal(n_pix, rng).astype(np.complex64)).to(dev)
            l, m = (pix % N - N // 2).double() * (fov / N), (pix // N - N // 2).double() * (fov / N)
            lmn = torch.stack([l, m, -(l * l + m * m) / (1 + torch.sqrt(1 - l * l - m * m))], 1)
            turns = uvw @ lmn.T
            turns = 2 * np.pi * (turns - torch.round(turns))
            e = torch.polar(torch.ones_like(turns), turns)
            image = torch.zeros(N * N, dtype=torch.complex64, device=dev)
            image[pix] = amp
            for i, (got, want) in enumerate([(p.degrid(image.reshape(N, N), uvw), e.conj() @ amp.to(e.dtype)),
                                             (p.grid(uvw, vis).ravel()[pix], e.T @ vis.to(e.dtype))]):
                err[i] += rel(got.to(e.dtype).cpu().numpy(), want.cpu().numpy()) ** 2
    print(Np, np.sqrt(err / 4))
    assert err[1] <= 1.05 ** 2 * err[0]
