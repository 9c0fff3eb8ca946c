"""The tap rule at its ties and far from the origin, and FP64 plans in several chunks of planes.

With a pixel of 2^-8 the visibilities are periodic in u and v with period 2^8 (every phase is a whole
turn), so a coordinate and the same one many periods away have the same taps, offsets and value.
"""
import numpy as np
import pytest
import torch

from gpu_helpers import case, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


@pytest.mark.parametrize("W", [4, 7])
def test_taps_are_periodic(dev, W):
    from paper_2101_11172_gb300.wstack import Plan
    N, fov = 64, 0.25                                     # l_j = j / 256; u' = u / 2 on N' = 128
    rng = np.random.default_rng(3)
    base = np.concatenate([np.arange(-6, 7), np.arange(-6, 7) + 0.5, rng.integers(-200, 200, 40) / 16.0])
    uvw = np.zeros((base.size, 3))
    uvw[:, 0], uvw[:, 1] = base, base[::-1]
    uvw[:, 2] = rng.uniform(-20, 20, base.size)
    image = (rng.normal(size=(N, N)) + 1j * rng.normal(size=(N, N))).astype(np.complex64)
    with Plan(N, 0.25, W, fov, -20.0, 20.0, device=dev) as p:
        t_img = torch.from_numpy(image).to(dev)
        v0 = p.degrid(t_img, torch.from_numpy(uvw).to(dev))
        assert torch.isfinite(torch.view_as_real(v0)).all() and float(v0.abs().max()) > 0
        for periods in (1, -1, 3, 1 << 20, -(1 << 20), 1 << 28, -(1 << 31), 1 << 33):
            far = uvw.copy()
            far[:, 0] += 256.0 * periods
            far[:, 1] -= 256.0 * periods
            assert torch.equal(p.degrid(t_img, torch.from_numpy(far).to(dev)), v0), periods


@pytest.mark.parametrize("W,chunk", [(3, 1), (12, 5), (14, 7)])
def test_fp64_chunks(dev, monkeypatch, W, chunk):
    from paper_2101_11172_gb300 import WS_FLAG_FP64
    from paper_2101_11172_gb300.wstack import Plan
    c = case(N=64, M=700, W=W, wfac=20.0, seed=W)
    out = []
    for planes in (0, chunk):
        if planes:
            monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(planes))
        with Plan(c["N"], c["x0"], W, c["fov"], c["w_min"], c["w_max"], flags=WS_FLAG_FP64, device=dev) as p:
            uvw = torch.from_numpy(c["uvw"]).to(dev)
            out.append((p.degrid(torch.from_numpy(c["image"]).to(dev), uvw).cpu().numpy(),
                        p.grid(uvw, torch.from_numpy(c["vis"]).to(dev)).cpu().numpy()))
    # the same terms, summed in another order: FP64 rounding
    assert rel(out[1][0], out[0][0]) < 1e-13 and rel(out[1][1], out[0][1]) < 1e-13
