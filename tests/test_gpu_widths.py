"""Whole-row tiles at widths other than 512, 1024, 2048 and 4096 (any multiple of 8 from 128 to 8192),
against the oracle: the narrowest and widest, widths whose rows take 1 to 8 warps and one or two
vectors per thread, ragged last tiles and chunks, one-row matrices, stacks, with and without momentum."""
import pytest
import torch

from paper_2607_19058_gb300 import skewadam as S
from paper_2607_19058_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

E, B = WL.TIER_EXPERT, WL.TIER_BACKBONE
#          rows, width: rows of half a warp; 64-row chunks; 2 warps a row; 5 of 8 warps; a partial last warp; 1 row side by side;
#          two vectors a thread, the second for few lanes; three quarters of the warps; the widest of 8 warps
SHAPES = [(2113, 128), (700, 200), (2113, 256), (1, 256), (700, 264), (333, 776), (517, 1032), (131, 1408), (9, 2040), (130, 2056), (257, 2880),
          (301, 3072), (5, 4088), (2049, 4088)]
# 16 warps a row tile (in a step without the others: see the planner's any_widths)
WIDE = [(1, 4104), (130, 4104), (77, 5632), (131, 7128), (1500, 8192)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


def _workload(shapes, eps=1e-30):
    """More than the 32 MiB of gradient from which these widths take row tiles (64 with an eps that may bind)."""
    specs = [WL.Spec(f"{'eb'[t]}{n}x{m}", (n, m), (E, B)[t], expert=k % 8 if t == 0 else -1)
             for k, (n, m) in enumerate(shapes) for t in (0, 1)]
    m0, m1 = (1536, 768) if shapes is SHAPES else (4800, 5000)
    specs += [WL.Spec("se", (3, 130, m0), E), WL.Spec("sb", (2, 67, m1), B)]
    if eps > 1e-12:
        specs.append(WL.Spec("more", (6000, 1400) if shapes is SHAPES else (1000, 4200), B))
    assert 2 * sum(torch.Size(s.shape).numel() for s in specs) >= (64 if eps > 1e-12 else 32) << 20
    return WL.Workload("widths", specs, WL.HP(), "toy", steps=3)


@pytest.mark.parametrize("shapes", [SHAPES, WIDE], ids=["to4096", "to8192"])
@pytest.mark.parametrize("hp", [{}, dict(eps=1e-8, lr=3e-4, weight_decay=0.05),
                                dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=0.05)],
                         ids=["eps1e-30", "paper", "clipped"])
def test_any_width_rows(shapes, hp):
    """eps = 1e-8 binds the clamp at step 1 (and d = 0.05 clips, so that every tensor takes phase B); experts
    5 to 7 have zero gradients on odd steps."""
    import parity
    h = parity.Harness(_workload(shapes, **{k: v for k, v in hp.items() if k == "eps"}), hp_override=hp)
    assert all(h.opt.route(k) == S.ROUTE_ROWS for k in range(len(h.wl.specs)))
    for t in range(1, 4):
        h.step(t, seed=17 * t, **({"gscale": 0.37} if t == 2 else {}))
    h.opt.sync_status()
    h.close()


# (16.8M elements are what takes such a matrix to row tiles when it is alone; the row sums of 4124839 x 1
# fill the no-alloc scratch; the last takes wide flat tiles)
@pytest.mark.parametrize("shape,tier", [((700, 264), E), ((12001, 1408), E), ((5601, 3072), B), ((2400, 7128), E),
                                        ((2051, 8192), B), ((4124839, 1), E), ((70, 10247), B)])
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
        S.skew_step_tensor_noalloc(w_na.data_ptr(), g.data_ptr(), 2, shape[0], shape[1], tier, 0, hp, state.data_ptr(),
                                   ref.state_bytes, 0, t, 1e-3, 77, torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        assert torch.equal(w_ref.view(torch.int16), w_na.view(torch.int16))
        assert torch.equal(ref.state[: ref.state_bytes].view(torch.float32), state)
    ref.close()
