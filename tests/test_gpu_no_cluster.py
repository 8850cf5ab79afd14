"""Where no thread-block cluster of the size asked for can be resident (here: the
answer of the occupancy query is injected on the host), a small formula is
contracted by a smaller cluster or level by level, and a batch without
clusters: the same counts."""
import pytest

from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()
    yield
    tnc.inject_failure("none")


@pytest.mark.parametrize("R", [1, 4, 7])
@pytest.mark.parametrize("n,smaller", [(80, True), (44, False)])  # packed for clusters of 16 CTAs and of 8
def test_small_formula(n, smaller, R):
    p = tnc.plan_formula(I.cubic_vertex_cover(n, 0), heuristic="best", rank_cap=32)
    want = tnc.contract_noalloc(p, n_residues=R)
    for broken in (False, True, False):
        if broken:
            tnc.inject_failure("cluster")
        r = tnc.contract(p, n_residues=R)
        assert r.residues.tolist() == want.residues.tolist() and r.counts == want.counts and r.flags == want.flags
        assert (tnc.last_launch_counts()["level"] == 1) == (smaller or not broken)


def test_batch():
    import torch
    sizes = (72, 72, 30, 24)
    plans = {n: tnc.plan_formula(I.cubic_vertex_cover(n, n), heuristic="gn") for n in sizes}
    tnc.inject_failure("cluster")
    b = tnc.Batch([plans[n] for n in sizes], n_residues=4)
    for shape in ((256, 0, 0), (128, 16384, 1)):
        b.set_launch(*shape)
        ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
        b.upload(ws)
        b.launch(ws)
        for n, r in zip(sizes, b.download(ws)):
            assert r.residues.tolist() == tnc.contract_noalloc(plans[n], n_residues=4).residues.tolist()
