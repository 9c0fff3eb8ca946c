"""The deterministic mode keeps each cell's fixed-point sum in two words, and every
addition to the low word carries into the high one: visibilities that occur once
with each sign leave sums of exactly zero, whatever their order."""
import numpy as np
import pytest

from gpu_helpers import case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


# N = 16: a grid so small that footprints wrap within a tile (N' = 32); W = 12: the widest footprint
@pytest.mark.parametrize("N,W,M,size", [(16, 7, 500, 1.0), (96, 4, 3000, 1.0), (64, 7, 4000, 1e-25),
                                        (64, 8, 4000, 1e25), (96, 12, 1500, 1.0)])
def test_opposite_visibilities_cancel_exactly(dev, N, W, M, size):
    from paper_2101_11172_gb300 import WS_FLAG_DETERMINISTIC
    from paper_2101_11172_gb300.wstack import Plan
    c = case(N=N, M=M, W=W, wfac=16.0, seed=11)
    order = np.random.default_rng(3).permutation(2 * M)
    uvw = np.concatenate([c["uvw"], c["uvw"]])[order]
    vis = np.concatenate([c["vis"], -c["vis"]])[order] * size
    with Plan(c["N"], c["x0"], c["W"], c["fov"], c["w_min"], c["w_max"], flags=WS_FLAG_DETERMINISTIC, device=dev) as p:
        u = torch.from_numpy(np.ascontiguousarray(uvw)).to(dev)
        v = torch.from_numpy(np.ascontiguousarray(vis)).to(torch.complex64).to(dev)
        d = p.grid(u, v)
        assert torch.count_nonzero(d).item() == 0
        one = p.grid(u[:M], v[:M])                       # no cancellation: finite, not zero
        assert torch.isfinite(torch.view_as_real(one)).all() and torch.count_nonzero(one).item() > 0
