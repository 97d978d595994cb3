"""Strip and flat tiles against the oracle: factored tensors without 16-byte row-vectors (odd widths
below and above 8, fp32, unaligned pointers, stacks whose matrices start inside a Philox block), at
both tile sizes (few strip-path elements, and many)."""
import pytest

from paper_2607_19058_gb300 import workloads as WL

pytestmark = pytest.mark.gpu

E, B, R = WL.TIER_EXPERT, WL.TIER_BACKBONE, WL.TIER_ROUTER


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_19058_gb300 import _build
    _build.build()
    import oracle
    oracle.build()


def _specs():
    shapes = [(1, 1), (3000, 1), (1025, 2), (700, 7), (257, 9), (1, 8191), (300, 127), (37, 333), (129, 1001), (513, 60),
              (70, 4100), (9, 5000)]
    out = [WL.Spec(f"{'eb'[t]}{n}x{m}{'f' if f else ''}", (n, m), (E, B)[t], expert=k % 8 if t == 0 else -1, fp32=f)
           for k, (n, m) in enumerate(shapes) for t in (0, 1) for f in (False, True)]
    out += [WL.Spec(f"s{k}x{n}x{m}", (k, n, m), t) for k, n, m, t in ((3, 5, 7, E), (5, 33, 13, B), (2, 3, 1, E))]
    return out + [WL.Spec("v4099", (4099,), B), WL.Spec("v4099f", (4099,), B, fp32=True), WL.Spec("r33x65", (33, 65), R),
                  WL.Spec("r3x33x65", (3, 33, 65), R)]


@pytest.mark.parametrize("many", [False, True], ids=["few", "many"])
@pytest.mark.parametrize("hp", [{}, dict(eps=1e-8, lr=3e-4, weight_decay=0.05)], ids=["eps1e-30", "paper"])
def test_flat_and_strip_tiles(many, hp):
    import parity
    specs = _specs()
    misalign = tuple(range(0, len(specs), 5))
    if many:  # past the line where strip tiles grow to 32 rows per thread
        specs += [WL.Spec("e4100x8200", (4100, 8200), E, expert=0), WL.Spec("b7001x901", (7001, 901), B)]
    h = parity.Harness(WL.Workload("strips", specs, WL.HP(), "toy", steps=2), hp_override=hp, misalign=misalign)
    for t in (1, 2):
        h.step(t, seed=23 * t, **({"gscale": 0.37} if t == 2 else {}))
    h.close()


@pytest.mark.parametrize("many", [False, True], ids=["few", "many"])
@pytest.mark.parametrize("hp", [{}, dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=0.05)], ids=["eps1e-30", "clip"])
def test_wide_flat_tiles(many, hp):
    """More columns than a tile's shared memory has room for: tiles of 1024 columns by 8 or (many) 64 rows, whose
    vectors straddle strips and rows; and the widest that need none. Last strips of 1, 7 and 1024 columns, one-row matrices, rows past a tile."""
    import parity
    shapes = [(5, 4095), (9, 4096), (7, 4097), (1, 8193), (5, 10241), (9, 10247), (66, 8450), (33, 50257), (4, 16384), (35, 9001)]
    specs = [WL.Spec(f"{'eb'[t]}{n}x{m}{'f' if f else ''}", (n, m), (E, B)[t], expert=k % 8 if t == 0 else -1, fp32=f)
             for k, (n, m) in enumerate(shapes) for t in (0, 1) for f in (False, True)]
    specs += [WL.Spec("s3x5x8201", (3, 5, 8201), E), WL.Spec("s2x9x10243", (2, 9, 10243), B)]
    misalign = tuple(range(0, len(specs), 3))
    if many:  # tiles grow to 64 rows
        specs.append(WL.Spec("e4100x8200", (4100, 8200), E, expert=0))
    h = parity.Harness(WL.Workload("wide", specs, WL.HP(), "toy", steps=2), hp_override=hp, misalign=misalign)
    for t in (1, 2):
        h.step(t, seed=31 * t, **({"gscale": 0.37} if t == 2 else {}))
    h.close()


@pytest.mark.parametrize("rows", [10007, 50007, 166669, 300007])
@pytest.mark.parametrize("hp", [{}, dict(eps=1e-8, lr=3e-4, weight_decay=0.05, clip_d=0.05)], ids=["eps1e-30", "clip"])
def test_tile_heights(rows, hp):
    """One matrix of 120 columns sets the step's strip elements (1.2M, 6M, 20M, 36M) and so the rows per strip tile (8,
    16, 32, 32 of each thread) and the rounds of a flat tile (4, 8, 16, 32), for 16-byte row-vectors of 3 to 31
    lanes a row and more, odd widths, fp32 and unaligned tensors beside it."""
    import parity
    shapes = [(1100, 24), (2100, 64), (257, 248), (300, 776), (33, 8200), (700, 7), (4100, 3), (129, 1001), (9, 4095), (70, 9001)]
    specs = [WL.Spec(f"{'eb'[t]}{n}x{m}{'f' if f else ''}", (n, m), (E, B)[t], fp32=f)
             for k, (n, m) in enumerate(shapes) for t, f in ((k % 2, False), (1 - k % 2, k % 3 == 0))]
    specs.append(WL.Spec(f"e{rows}x120", (rows, 120), (E, B)[rows % 2]))
    h = parity.Harness(WL.Workload("heights", specs, WL.HP(), "toy", steps=2), hp_override=hp, misalign=tuple(range(0, len(specs) - 1, 4)))
    for t in (1, 2):
        h.step(t, seed=37 * t, **({"gscale": 0.37} if t == 2 else {}))
    h.close()
