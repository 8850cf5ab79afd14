"""A formula with descriptors of nearly a CTA's shared memory is accepted in a
batch whether it is contracted by one CTA or, as the batch's heavy formula, by
a cluster, whose finer segments take a little more descriptors."""
import pytest

from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


def _union(forms):
    clauses, kinds, n = [], [], 0
    for f in forms:
        clauses += [tuple(v + n for v in vs) for vs in f.clauses]
        kinds += list(f.kinds)
        n += f.n_vars
    return I.Formula(n, clauses, kinds)


def _accepted(plans):
    try:
        return tnc.Batch(plans, n_residues=2)
    except tnc.TncError as e:
        assert e.code == -2
        return None


def test_heavy_formula_is_accepted_where_a_light_one_is():
    import torch
    core = [I.cubic_vertex_cover(70, 0)] + [I.cubic_vertex_cover(60, s) for s in range(17)]
    pair = I.Formula(2, [(0, 1)], [I.KIND_OR])
    # 40 formulas at least as heavy: the one beside them is not heavier than the batch's average
    heavier = [tnc.plan_formula(I.cubic_vertex_cover(110, 0), heuristic="best", rank_cap=24)] * 40
    seen, largest = set(), None
    for n in range(84, 110, 2):  # 92 bytes of descriptors a pair, the whole around 227 KiB
        p = tnc.plan_formula(_union(core + [pair] * n), heuristic="greedy", rank_cap=24)
        light, heavy = _accepted(heavier + [p]), _accepted([p])
        assert (light is None) == (heavy is None), n
        seen.add(heavy is None)
        if heavy is not None:
            largest = (p, heavy)
    assert seen == {True, False}  # the limit lies within the sizes tried
    p, b = largest
    ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
    b.upload(ws)
    b.launch(ws)
    assert b.download(ws)[0].residues.tolist() == tnc.contract(p, n_residues=2).residues.tolist()
