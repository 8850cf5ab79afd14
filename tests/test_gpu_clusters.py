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
