"""The same tensors on every route a step may take them: the single launch of small tensors, strip and
flat tiles in launches of their own, the same riding beside row tiles, and row tiles; under every policy,
with the gradient scale and both eps. What decides is what else the step holds."""
import pytest

from paper_2607_19058_gb300 import skewadam as S
from paper_2607_19058_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

E, B = WL.TIER_EXPERT, WL.TIER_BACKBONE


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


BESIDE = {"small": [], "own": [WL.Spec("e10007x120", (10007, 120), E)],
          "riding": [WL.Spec("e10007x120", (10007, 120), E), WL.Spec("e2100x4096", (2100, 4096), E)]}
ROUTE = {"small": S.ROUTE_SMALL, "own": S.ROUTE_OWN, "riding": S.ROUTE_RIDING}


@pytest.mark.parametrize("beside", list(BESIDE))
@pytest.mark.parametrize("hp", [dict(policy=p) for p in range(5)] + [dict(eps=1e-8, lr=3e-4, weight_decay=0.05)],
                         ids=["tiered", "expert_momentum", "factored_router", "uniform", "adafactor", "paper"])
def test_toy_set(beside, hp):
    """The toy set (fp32 router and norms), zero-gradient experts at t = 1, gamma = 0.37 at t = 2."""
    import parity
    toy = WL.toy_fp32().specs
    specs = list(toy) + BESIDE[beside]
    h = parity.Harness(WL.Workload("routes", specs, WL.HP(**{k: v for k, v in hp.items() if k == "policy"}), "toy", steps=3),
                       hp_override=hp)
    assert {h.opt.route(k) for k in range(len(toy))} == {ROUTE[beside]}
    for t in (1, 2, 3):
        h.step(t, seed=41 * t, **({"gscale": 0.37} if t == 2 else {}))
    h.opt.sync_status()
    h.close()


@pytest.mark.parametrize("policy", [WL.POLICY_TIERED, WL.POLICY_EXPERT_MOMENTUM])
def test_tiny_matrices_on_row_tiles(policy):
    """Matrices of fewer rows than one chunk of a row tile (1 to 5 rows; a stack of one-row matrices), with
    and without momentum, beside one that is too large for the single launch."""
    import parity
    specs = [WL.Spec(f"{'eb'[t]}{n}x{m}", (n, m), (E, B)[t], expert=k if t == 0 else -1)
             for k, (n, m) in enumerate([(1, 4096), (2, 1024), (3, 512), (5, 2048), (1, 520), (3, 4088)]) for t in (0, 1)]
    specs += [WL.Spec("s3x1x1024", (3, 1, 1024), E), WL.Spec("e4500x4096", (4500, 4096), E)]
    h = parity.Harness(WL.Workload("tiny_rows", specs, WL.HP(policy=policy), "normal", steps=3))
    assert all(h.opt.route(k) == S.ROUTE_ROWS for k in range(len(specs)))
    for t in (1, 2, 3):
        h.step(t, seed=43 * t)
    h.opt.sync_status()
    h.close()
