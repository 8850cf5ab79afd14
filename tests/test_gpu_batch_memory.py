"""Device memory of a batch: no more arena slots than formulas (or resident
CTAs), also where clusters of CTAs contract the heavy formulas, and the light
ones share what slots there are."""
import pytest

from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


@pytest.mark.parametrize("R", [1, 4])
@pytest.mark.parametrize("sizes", [
    (72,) * 19 + (30,),        # fewer light formulas than CTAs: most CTAs find no slot
    (72,) * 3 + (30,) * 5,
    (72, 30),
    (72,) + (24,) * 700,       # more light formulas than CTAs
    (70,) * 90 + (30,) * 90,   # more heavy formulas than clusters
])
def test_batch_memory_is_a_slot_per_formula(sizes, R):
    import torch
    plans = {n: tnc.plan_formula(I.cubic_vertex_cover(n, n), heuristic="gn") for n in set(sizes)}
    want = {n: tnc.contract_noalloc(p, n_residues=R) for n, p in plans.items()}
    b = tnc.Batch([plans[n] for n in sizes], n_residues=R)
    largest = max(p.stats.batch_arena_entries for p in plans.values()) + 7
    limbs = (31 * R + 31) // 32
    rest = b.info()[0] + len(sizes) * 4 * (R + limbs) + 4096  # descriptors, results; sections aligned
    assert b.workspace_bytes() <= rest + len(sizes) * largest * 4 * R
    ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
    b.upload(ws)
    for shape in ((256, 0, 0), (64, 0, 0), (128, 16384, 1)):
        b.set_launch(*shape)
        b.launch(ws)
        for n, r in zip(sizes, b.download(ws)):
            assert r.residues.tolist() == want[n].residues.tolist() and r.counts == want[n].counts, (n, shape)


def test_deep_formulas_beside_heavy_ones():
    """Formulas of many levels are light even where smaller, flatter ones are heavy."""
    import torch
    forms = [I.cubic_vertex_cover(72, 72), I.one_in_three(70, 43, 25), I.cubic_vertex_cover(50, 14), I.cubic_vertex_cover(24, 0)]
    plans = [tnc.plan_formula(f, heuristic="gn", rank_cap=24) for f in forms]
    work = [p.stats.total_macs + p.stats.total_entries for p in plans]
    per_level = [w / p.stats.depth for w, p in zip(work, plans)]
    assert work[1] > work[2] and per_level[1] < 5500 < per_level[2]
    b = tnc.Batch(plans, n_residues=2)
    ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
    b.upload(ws)
    b.launch(ws)
    for p, r in zip(plans, b.download(ws)):
        assert r.residues.tolist() == tnc.contract_noalloc(p, n_residues=2).residues.tolist()


def test_three_residues_take_four_only_where_that_is_small():
    """Launches (residue groups and the CRT) and device memory of 3 residues."""
    small = tnc.plan_formula(I.cubic_vertex_cover(72, 72), heuristic="gn")
    large = tnc.plan_formula(I.cubic_vertex_cover(110, 0), heuristic="best", rank_cap=24)
    assert tnc.Batch([small], n_residues=3).info()[3] == 2       # one group of four
    assert tnc.Batch([small, large], n_residues=3).info()[3] == 3  # two and one
    b = tnc.Batch([small] * 6000, n_residues=3)  # arenas beyond 1 GiB with four
    assert b.info()[3] == 3
    rest = b.info()[0] + 6000 * 4 * (3 + 3) + 4096
    assert b.workspace_bytes() <= rest + 6000 * (small.stats.batch_arena_entries + 7) * 4 * 2


def test_graph_replays_with_heavy_formulas():
    """On a stream of its own the launch is a captured graph: its counters start anew each time."""
    import torch
    sizes = (72, 72, 30, 24, 24)
    plans = {n: tnc.plan_formula(I.cubic_vertex_cover(n, n), heuristic="gn") for n in sizes}
    want = [tnc.contract_noalloc(plans[n], n_residues=4).residues.tolist() for n in sizes]
    b = tnc.Batch([plans[n] for n in sizes], n_residues=4)
    ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    st = torch.cuda.Stream()
    b.upload(ws, st)
    for _ in range(3):
        b.launch(ws, st)
        assert [r.residues.tolist() for r in b.download(ws, st)] == want
