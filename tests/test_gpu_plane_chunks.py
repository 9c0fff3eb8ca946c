"""What a call gives when its planes come in several chunks (little free memory, a batch's slice)."""
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


def _case(N, M, w_half, seed, fov=0.2):
    rng = synth.rng_for(0, 9000 + seed)
    uvw = synth.disc_uvw(M, 0.45 * N / fov, w_half, rng)
    return dict(N=N, fov=fov, uvw=uvw, vis=synth.complex_normal(M, rng), w_min=float(uvw[:, 2].min()),
                w_max=float(uvw[:, 2].max()))


def _plan(c, dev, W=7, x0=0.25, flags=0):
    from paper_2101_11172_gb300.wstack import Plan
    return Plan(c["N"], x0, W, c["fov"], c["w_min"], c["w_max"], flags=flags, device=dev)


def _inputs(c, dev):
    return torch.from_numpy(c["uvw"]).to(dev), torch.from_numpy(c["vis"]).to(torch.complex64).to(dev)


@pytest.mark.parametrize("N,W,x0", [(64, 7, 0.25), (200, 10, 0.25), (256, 7, 0.25), (512, 4, 0.375)])
def test_deterministic_image_does_not_depend_on_the_chunks(dev, monkeypatch, N, W, x0):
    """Bit for bit, over chunks of 8 planes up to all of them and in a batch's small slice."""
    from paper_2101_11172_gb300 import WS_FLAG_DETERMINISTIC
    from paper_2101_11172_gb300.batch import Batch
    c = _case(N, 3000, 6000.0 * x0, N)              # 67 planes
    uvw, vis = _inputs(c, dev)
    images = []
    for chunk in (0, 8, 24, 64):
        if chunk:
            monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(chunk))
        with _plan(c, dev, W, x0, WS_FLAG_DETERMINISTIC) as p:
            assert p.Nw > 64 and (p.planes_per_chunk == chunk or not chunk)
            images.append(p.grid(uvw, vis))
            Np = p.Np
    with Batch([(N, c["fov"], c["w_min"], c["w_max"], 3000)], x0, W, branches=1, workspace_bytes=17 * Np * Np * 8,
               flags=WS_FLAG_DETERMINISTIC, device=dev) as b:
        images += b.grid([uvw], [vis])
    for d in images[1:]:
        assert torch.equal(d, images[0])


@pytest.mark.parametrize("planes", [9, 17, 40])
def test_batch_in_a_small_slice(dev, planes):
    """Rows shared by no more CTAs than a chunk has planes give the plan's image to summation order."""
    from paper_2101_11172_gb300.batch import Batch
    c = _case(128, 3000, 1500.0, planes)
    uvw, vis = _inputs(c, dev)
    with _plan(c, dev) as p:
        assert p.Nw > 60
        whole, Np = p.grid(uvw, vis), p.Np
    with Batch([(128, c["fov"], c["w_min"], c["w_max"], 3000)], 0.25, 7, branches=1,
               workspace_bytes=planes * Np * Np * 8, device=dev) as b:
        for _ in range(2):
            assert rel(b.grid([uvw], [vis])[0].cpu().numpy(), whole.cpu().numpy()) < 1e-6


@pytest.mark.parametrize("N,chunk,flags", [(64, 0, 0), (64, 24, 0), (200, 16, 0), (256, 24, 1 << 6)])
def test_incomplete_rows_count_once(dev, monkeypatch, N, chunk, flags):
    """Waits that give up at once (host knob, every copy still lands) in rows shared by several CTAs and
    planes in several chunks: one count per row, no row written, and the next call is complete."""
    from paper_2101_11172_gb300 import _lib
    c = _case(N, 3000, 1500.0, N + chunk)
    uvw, vis = _inputs(c, dev)
    if chunk:
        monkeypatch.setenv("WS_PLANES_PER_CHUNK", str(chunk))
    with _plan(c, dev, flags=flags) as p:
        assert p.Nw > 60
        want = p.grid(uvw, vis)
        p.stats(reset=True)
        out = torch.full_like(want, 7.0)
        monkeypatch.setenv("WS_WAIT_POLLS", "0")
        with pytest.raises(_lib.WsError) as err:
            p.grid(uvw, vis, out=out)
        assert err.value.status == _lib.WS_ERR_TIMEOUT
        assert p.stats(reset=True)["waits_timed_out"] == N
        assert bool((out == 7.0).all())
        monkeypatch.delenv("WS_WAIT_POLLS")
        assert rel(p.grid(uvw, vis, out=out).cpu().numpy(), want.cpu().numpy()) < 1e-6
        assert p.stats()["waits_timed_out"] == 0


def test_new_plans_on_a_stream_of_their_own(dev):
    """A plan's first call, on a stream that is not ordered after the default one, finds its row counters cleared."""
    c = _case(64, 3000, 1500.0, 3)
    uvw, vis = _inputs(c, dev)
    with _plan(c, dev) as p:
        want = p.grid(uvw, vis).cpu().numpy()
    side = torch.cuda.Stream(dev)
    side.wait_stream(torch.cuda.current_stream(dev))
    for _ in range(20):
        torch.cuda.empty_cache()                       # the next plan's buffers may be memory that held anything
        with _plan(c, dev) as p, torch.cuda.stream(side):
            out = torch.zeros(64, 64, dtype=torch.complex64, device=dev)
            p.grid(uvw, vis, out=out)
            side.synchronize()
            assert rel(out.cpu().numpy(), want) < 1e-6
