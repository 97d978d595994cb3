"""A step captured into a CUDA graph replays to the same weights and state as direct calls (the
launches of a step are programmatic dependents of one another), on a side stream and with work of
the caller's before and after it."""
import pytest
import torch

from paper_2607_19058_gb300 import skewadam as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()


SHAPES = [((300, 4096), 0), ((517, 776), 1), ((64, 128), 1), ((40, 13), 0), ((1000,), 0), ((128, 64), 2)]


def _set(seed, shapes):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    ps = []
    for shape, tier in shapes:
        w = torch.empty(shape, device="cuda").normal_(0, 0.02, generator=g).to(torch.bfloat16)
        ps.append((w, torch.empty(shape, device="cuda").normal_(0, 1e-3, generator=g).to(torch.bfloat16), tier))
    return ps, S.SkewAdam(ps, S.hparams(eps=1e-30))


# row tiles with strip and flat tiles beside them; strip and flat tiles alone; the single launch of small tensors
@pytest.mark.parametrize("shapes,launches", [(SHAPES, 5), (SHAPES[2:] + [((9000, 64), 0), ((8000, 72), 1), ((20000, 41), 0)], 5), (SHAPES[2:], 1)],
                         ids=["rows", "light", "small"])
def test_captured_step_equals_direct(shapes, launches):
    pa, a = _set(1, shapes)
    pb, b = _set(1, shapes)
    assert S.skew_launches_per_step(b.h) == launches
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        b.step(1, 1e-3, 7)           # loads the kernels before the capture
    a.step(1, 1e-3, 7)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        for _, g, _ in pb:
            g.mul_(0.5)
        b.step(2, 1e-3, 7)
        for _, g, _ in pb:
            g.mul_(2.0)
    for _ in range(3):
        for _, g, _ in pa:
            g.mul_(0.5)
        a.step(2, 1e-3, 7)
        for _, g, _ in pa:
            g.mul_(2.0)
        graph.replay()
    torch.cuda.synchronize()
    a.sync_status()
    b.sync_status()
    for (wa, _, _), (wb, _, _) in zip(pa, pb):
        assert torch.equal(wa.view(torch.int16), wb.view(torch.int16))
    assert torch.equal(a.state, b.state)
