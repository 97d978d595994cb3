"""Steps of small tensors only, which run as one launch (a cluster of CTAs per tensor), against the
oracle: cluster sizes 1, 2 and 8, slices with no rows, one-row and one-column matrices, every kind and
dtype, unaligned pointers, stacks, the clip factor, a zero gradient, the clamp."""
import pytest
import torch

from paper_2607_19058_gb300 import skewadam as S
from paper_2607_19058_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

E, B, R = WL.TIER_EXPERT, WL.TIER_BACKBONE, WL.TIER_ROUTER


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


def _specs(shapes):
    out = [WL.Spec(f"{'eb'[t]}{n}x{m}{'f' if f else ''}", (n, m), (E, B)[t], expert=k % 8 if t == 0 else -1, fp32=f)
           for k, (n, m) in enumerate(shapes) for t in (0, 1) for f in (False, True)]
    return out + [WL.Spec("s3x5x7", (3, 5, 7), E), WL.Spec("s2x33x13", (2, 33, 13), B), WL.Spec("v4099", (4099,), B),
                  WL.Spec("v7f", (7,), B, fp32=True), WL.Spec("r33x65", (33, 65), R), WL.Spec("r64x8f", (64, 8), R, fp32=True)]


@pytest.mark.parametrize("shapes", [
    [(1, 1), (1, 4096), (3000, 1), (64, 31), (63, 64), (129, 128), (5, 1000)],        # few elements: larger clusters
    [(512, 64), (200, 208), (47, 1000), (9, 5000), (700, 60), (1023, 33), (40000, 1)] * 4,  # one CTA a tensor
    [(640, 640), (8, 4000), (300, 1001)],                                              # slices of clusters of eight
], ids=["tiny", "many", "clusters"])
@pytest.mark.parametrize("hp", [{}, dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=0.05)], ids=["eps1e-30", "clip"])
def test_small_step(shapes, hp):
    import parity
    specs = _specs(shapes)
    h = parity.Harness(WL.Workload("small", specs, WL.HP(), "toy", steps=3), hp_override=hp,
                       misalign=tuple(range(0, len(specs), 5)))
    assert S.skew_launches_per_step(h.opt.h) == 1
    for t in range(1, 4):
        h.load_grads(t)
        if t == 1:
            h.G[1].zero_()
        h.step(t, seed=29 * t, grads_loaded=True, **({"gscale": 0.37} if t == 2 else {}))
    h.opt.sync_status()
    h.close()


@pytest.mark.parametrize("shape,tier", [((141, 208), E), ((512, 64), B), ((4096,), B), ((64, 127), R), ((700, 500), E)])
def test_noalloc_matches_the_handle(shape, tier):
    torch.manual_seed(0)
    w0 = (torch.randn(shape, device="cuda") * 0.02).to(torch.bfloat16)
    g = torch.empty(shape, dtype=torch.bfloat16, device="cuda")
    hp = S.hparams(0.9, 0.999, 1e-30, 1.0, 0.1, S.POLICY_TIERED)
    w_ref, w_na = w0.clone(), w0.clone()
    ref = S.SkewAdam([(w_ref, g, tier)], hp)
    state = torch.zeros(ref.state_bytes // 4, dtype=torch.float32, device="cuda")
    for t in (1, 2):
        g.copy_((torch.randn(shape, device="cuda") * 1e-3).to(torch.bfloat16))
        ref.step(t, 1e-3, 77)
        S.skew_step_tensor_noalloc(w_na.data_ptr(), g.data_ptr(), len(shape), shape[0], shape[1] if len(shape) == 2 else 0,
                                   tier, 0, hp, state.data_ptr(), ref.state_bytes, 0, t, 1e-3, 77,
                                   torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(w_ref.view(torch.int16), w_na.view(torch.int16))
        assert torch.equal(ref.state[: ref.state_bytes].view(torch.float32), state)
    ref.close()
