"""Formulas contracted by whole clusters: the heavy ones of a batch.

Counts are exact integers, so the tolerance is zero: every residue of the
batch equals the single-formula contraction's, and a sample the oracle's."""
import pytest

import oracle
from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu

WIDE = [2147483647, 2147483629, 2147483587, 2147483579, 2147483563]


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


@pytest.mark.parametrize("R,wide", [(1, False), (2, True), (3, False), (4, False), (5, True)])
@pytest.mark.parametrize("sizes", [
    (76, 20, 40, 12, 64),           # heavy formulas and light ones
    (64, 66, 68),                   # all heavy: fewer formulas than clusters
    (72,) + (24,) * 700,            # one heavy formula, more light ones than resident CTAs
    (70,) * 90 + (30,) * 90,        # more heavy formulas than clusters at once
])
def test_batch_with_heavy_formulas(sizes, R, wide):
    import torch
    kinds = sorted(set(sizes))
    forms = {}
    for n in kinds:
        f = I.cubic_vertex_cover(n, n)
        if n == 64:
            f.open_vars = [3, 40, 11]
        forms[n] = f
    one = {n: tnc.plan_formula(f, heuristic="gn") for n, f in forms.items()}
    plans = [one[n] for n in sizes]
    primes = WIDE[:R] if wide else None
    b = tnc.Batch(plans, n_residues=R, primes=primes)
    ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
    want = {n: tnc.contract(one[n], n_residues=R, primes=primes) for n in kinds}
    for n in kinds:
        if n <= 40:
            assert want[n].residues.tolist() == oracle.residues(oracle.count(forms[n]), want[n].primes)
    b.upload(ws)
    for shape in ((256, 0, 0), (64, 16384, 0), (128, 0, 1)):
        b.set_launch(*shape)
        b.launch(ws)
        got = b.download(ws)
        for n, r in zip(sizes, got):
            assert r.residues.tolist() == want[n].residues.tolist() and r.counts == want[n].counts, (n, shape)


def _solo_forms():
    open_vc = I.cubic_vertex_cover(30, 3)
    open_vc.open_vars = [7, 0, 12, 29, 4]
    return {"one_variable": I.Formula(1, [], []), "worked_example": I.worked_example(),
            "1in3_n20": I.one_in_three(20, 12, 3), "open_vc_n30": open_vc, "vc_n44": I.cubic_vertex_cover(44, 0),
            "vc_n60": I.cubic_vertex_cover(60, 0), "vc_n90": I.cubic_vertex_cover(90, 1)}


@pytest.mark.parametrize("R,wide", [(1, False), (2, True), (3, False), (4, False), (5, True), (7, False), (16, False)])
@pytest.mark.parametrize("name", list(_solo_forms()))
def test_one_launch_contraction(name, R, wide):
    """Small formulas run in one launch per residue group; the allocation-free
    entry point runs the same plan step by step."""
    f = _solo_forms()[name]
    p = tnc.plan_formula(f, heuristic="best")
    primes = WIDE[:R] if wide else None
    want = tnc.contract_noalloc(p, n_residues=R, primes=primes)
    for _ in range(2):
        r = tnc.contract(p, n_residues=R, primes=primes)
        lc = tnc.last_launch_counts()
        assert lc["level"] == 1 and lc["crt"] == 1 and lc["grid_step"] == lc["outer"] == 0
        assert r.residues.tolist() == want.residues.tolist() and r.counts == want.counts and r.flags == want.flags
    if f.n_vars <= 60:
        assert r.residues.tolist() == oracle.residues(oracle.count(f), r.primes)
