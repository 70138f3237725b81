"""The plain calls away from ordinary scenes: more views under capture than in
the calls before it."""
import pytest

from paper_2606_09074_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2606_09074_gb300 import binding as rb
    return torch, rb, torch.device("cuda", 0)


def uploaded(torch, rb, dev, w):
    return torch.from_numpy(w.scene.pos).to(dev), torch.from_numpy(w.scene.attr).to(dev), rb.cameras_to_device(w.cams, dev)


@pytest.mark.parametrize("n", [100_000, 300_000])
def test_capture_with_more_views_than_before(env, n):
    """A captured call may score more views than the calls that sized the
    scratch: what they left holds its scene scratch (512 camera records more
    are 56 KB), and its scores have the bits of an uncaptured call."""
    torch, rb, dev = env
    pos, attr, cams = uploaded(torch, rb, dev, synth.random_scene(seed=n, n=n, v=512, means="core_shell"))
    ref = rb.Context(0)
    want = ref.score(pos, attr, cams)
    torch.cuda.synchronize()
    ctx, stream = rb.Context(0), torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx.score(pos, attr, cams, n_views=64)
        stream.synchronize()
        out = torch.zeros(n, device=dev)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            ctx.score(pos, attr, cams, scores=out)
        for _ in range(2):
            graph.replay()
        stream.synchronize()
        assert torch.equal(out.view(torch.int32), want.view(torch.int32))
        ctx.check()
    ctx.close()
    ref.close()
