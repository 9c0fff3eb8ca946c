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
