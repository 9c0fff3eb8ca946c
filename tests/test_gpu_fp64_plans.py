"""Several FP64 plans alive at once, and the memory they take."""
import pytest
import torch

from gpu_helpers import case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return torch.device("cuda", 0)


def _plan(c, dev):
    from paper_2101_11172_gb300 import WS_FLAG_FP64
    from paper_2101_11172_gb300.wstack import Plan
    return Plan(c["N"], c["x0"], c["W"], c["fov"], c["w_min"], c["w_max"], flags=WS_FLAG_FP64, device=dev)


def _both(p, c, dev):
    uvw = torch.from_numpy(c["uvw"]).to(dev)
    return p.degrid(torch.from_numpy(c["image"]).to(dev), uvw), p.grid(uvw, torch.from_numpy(c["vis"]).to(dev))


# N' = 32 .. 2048: 16 lines and one or two per CTA, 8 to 64 KB of shared memory
@pytest.mark.parametrize("first,second", [(128, 64), (128, 16), (1024, 32), (64, 512)])
def test_a_second_plan_leaves_the_first_usable(dev, first, second):
    cs = [case(N=n, M=300, W=6, wfac=2.0, seed=n) for n in (first, second)]
    with _plan(cs[0], dev) as a:
        before = _both(a, cs[0], dev)
        with _plan(cs[1], dev) as b:
            _both(b, cs[1], dev)
            again = _both(a, cs[0], dev)
    for x, y in zip(before, again):                    # gridding sums with FP64 atomics
        assert torch.linalg.norm(x - y) <= 1e-13 * torch.linalg.norm(x)


def test_planes_stay_within_the_memory_budget(dev, monkeypatch):
    """WS_STACK_BYTES bounds the chunk of planes down to one, and the result does not depend on it."""
    c = case(N=128, M=300, W=6, wfac=16.0, seed=5)
    plane = (2 * c["N"]) ** 2 * 16
    out, used = [], []
    for planes in (0, 5, 0.5):
        if planes:
            monkeypatch.setenv("WS_STACK_BYTES", str(int(planes * plane)))
        with _plan(c, dev) as p:
            used.append(p.workspace_bytes)
            out.append(_both(p, c, dev))
            assert p.Nw > 8
    assert used[0] - used[1] == (p.Nw - 5) * plane and used[0] - used[2] == (p.Nw - 1) * plane
    for o in out[1:]:
        for x, y in zip(out[0], o):                    # the same terms, summed in another order
            assert torch.linalg.norm(x - y) <= 1e-13 * torch.linalg.norm(x)
