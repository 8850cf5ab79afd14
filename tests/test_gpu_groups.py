"""Groups of formulas whose steps of one kind share launches: more plans than
one extraction takes (64), more dense steps of a tile width than one GEMM
launch takes (256), split-K steps of several plans, residue passes of 4, 2 and
1.  Exact integers: every count equals the same plan's contracted alone, and
one of each kind the oracle's."""
import pytest

import oracle
from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


@pytest.mark.parametrize("path,R,copies", [("tc_p8", 7, 100), ("tc_p8", 5, 1), ("int64", 3, 25), ("tc", 2, 17), ("tc", 7, 30)])
def test_group_equals_one_by_one(path, R, copies):
    forms = [I.cubic_vertex_cover(70, 0), I.cubic_vertex_cover(90, 4), I.cubic_vertex_cover(20, 1)]
    forms[2].open_vars = [2, 9]
    plans = [tnc.plan_formula(f, heuristic=h) for f, h in zip(forms, ("greedy", "bisect", "greedy"))]
    want = [tnc.contract_many([p, plans[2]], n_residues=R, path=path)[0] for p in plans]
    got = tnc.contract_many(plans * copies, n_residues=R, path=path, group=3 * copies)
    lc = tnc.last_launch_counts()
    assert lc["crt"] == 1 and lc["extract"] >= (3 * copies + 63) // 64
    if path == "tc_p8":
        assert lc["p8_gemm"] >= 3 * copies
    for i, r in enumerate(got):
        assert r.residues.tolist() == want[i % 3].residues.tolist() and r.counts == want[i % 3].counts, i
    for f, w in zip(forms[::2], want[::2]):
        assert w.residues.tolist() == oracle.residues(oracle.count(f, max_rank=28), w.primes)


@pytest.mark.parametrize("path,R", [("int64", 7), ("tc", 7), ("tc_p8", 11)])
def test_workspaces(path, R):
    """One workspace serves both u32 paths; less than the library would use, down to
    one residue group at a time, gives the same counts; too little is refused."""
    import torch
    f = I.cubic_vertex_cover(90, 4)
    p = tnc.plan_formula(f, heuristic="bisect", rank_cap=24)
    nb = tnc.workspace_bytes(p, R, "tc_p8" if path == "tc_p8" else "int64")
    want = tnc.contract(p, n_residues=R, path=path, workspace=torch.empty(nb, dtype=torch.uint8, device="cuda"))
    assert want.residues.tolist() == oracle.residues(oracle.count(f, max_rank=24), want.primes)
    ran = 0
    for k in range(1, 8):
        try:
            r = tnc.contract(p, n_residues=R, path=path, workspace=torch.empty(nb * k // 8, dtype=torch.uint8, device="cuda"))
        except ValueError:
            continue
        ran += 1
        assert r.residues.tolist() == want.residues.tolist() and r.counts == want.counts
    assert ran >= 1
    with pytest.raises(ValueError):
        tnc.contract(p, n_residues=R, path=path, workspace=torch.empty(4096, dtype=torch.uint8, device="cuda"))
