"""Row-path tensors whose eps clamp binds (eps = 1e-8, App. A), on both routes to sum(U^2): summed in
phase C where a bound proves that the update is not clipped (d = 1), and by phase B where it may be
(d = 0.05). Weights, state and the scalars (sum(U^2), RMS, clip factor) against the oracle; whole and
half phase-C tiles, last tiles without a second half, one-row matrices, stacks, zero-gradient experts."""
import pytest
import torch

from paper_2607_19058_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

E, B = WL.TIER_EXPERT, WL.TIER_BACKBONE


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


BILINEAR, PHASE_B, PHASE_C = 0, 1, 2


def _sum_from(opt):
    """Where the last step took each matrix's sum(U^2) from: the word at byte 52 of its 64-byte scalars, with which
    the workspace starts."""
    count = sum(max(1, opt.info(k).stack) for k in range(len(opt.params)))
    return opt.workspace[: 64 * count].cpu().view(torch.int32).view(count, 16)[:, 13].tolist()


@pytest.mark.parametrize("clip_d", [1.0, 0.05])
def test_clamped_tensors(clip_d):
    import parity
    specs = [WL.Spec("e301x4096", (301, 4096), E, expert=0), WL.Spec("b301x4096", (301, 4096), B),
             WL.Spec("e1x4096", (1, 4096), E, expert=1), WL.Spec("b2101x512", (2101, 512), B),
             WL.Spec("e2049x1024", (2049, 1024), E, expert=5), WL.Spec("s3x70x2048", (3, 70, 2048), E),
             WL.Spec("e2300x4096", (2300, 4096), E, expert=6)]
    h = parity.Harness(WL.Workload("clamp", specs, WL.HP(), "toy", steps=3),
                       hp_override=dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=clip_d))
    for t in range(1, 4):
        rep = h.step(t, seed=5 * t, **({"gscale": 0.37} if t == 2 else {}))
        assert (rep.clipped > 0) == (clip_d < 1.0)
        for src, where in zip(_sum_from(h.opt), [sp for sp in specs for _ in range(sp.shape[0] if len(sp.shape) == 3 else 1)]):
            if t % 2 and where.expert >= 5:
                assert src == BILINEAR, where      # no gradient
            elif clip_d < 1.0:
                assert src == PHASE_B, where
            elif t > 1 or where.tier == E:
                assert src == PHASE_C, where       # (momentum's first step is near d: either)
    h.opt.sync_status()
    h.close()


def test_more_queued_matrices_than_a_cta_reads_at_once():
    """300 matrices whose update is clipped (d = 0.05), queued for phase B: k_fallback reads its queue 256 at a
    time; one to five phase-C tiles each, with and without momentum, fixed and general widths, a stack."""
    import parity
    shapes = [(40, 512), (1100, 512), (70, 2048), (300, 776), (5, 4096), (600, 1032)]
    specs = [WL.Spec(f"{'eb'[k % 2]}{k}", shapes[k % 6], (E, B)[k % 2], expert=k % 5 if k % 2 == 0 else -1) for k in range(240)]
    specs.append(WL.Spec("s60x33x1024", (60, 33, 1024), E))
    h = parity.Harness(WL.Workload("queue", specs, WL.HP(), "toy", steps=2),
                       hp_override=dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=0.05))
    for t in (1, 2):
        assert h.step(t, seed=7 * t).clipped > 256
    h.opt.sync_status()
    h.close()
