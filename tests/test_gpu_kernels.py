"""Which kernels a contraction launches (tnc_last_kernel_launches), and their counts.

One step of 2^fa x 2^fb outputs and 2^k shared values decides the kernel: the
formula has k inner variables x_i, each in a weighted clause with some of the
fa open variables a and one with some of the b.  The last step of the order
contracts the two sides; its entries are prod_i sum_x T_i(x, a) U_i(x, b),
computed here modulo each prime in integers: the tolerance is zero."""
import random

import numpy as np
import pytest

import oracle
from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu

WIDE = [2147483647, 2147483629, 2147483587, 2147483579]


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


def _split(n, k, i):
    """Of n variables those of the i-th of k clauses (each in one; some clauses share where k > n)."""
    return list(range(i, n, k)) or [i % n]


def _formula(fa, fb, k, seed):
    rng = random.Random(seed)
    sides, tables = [], []
    for n, first in ((fa, k), (fb, k + fa)):
        for i in range(k):
            vs = _split(n, k, i)
            sides.append(tuple([i] + [first + v for v in vs]))
            tables.append([rng.getrandbits(32) for _ in range(2 << len(vs))])
    n_vars = k + fa + fb
    f = I.Formula(n_vars, sides, [I.KIND_TABLE] * (2 * k), tables, open_vars=list(range(k, n_vars)))
    nxt, order = 2 * k + n_vars, []

    def chain(ids):
        nonlocal nxt
        acc = ids[0]
        for j in ids[1:]:
            order.append((acc, j))
            acc, nxt = nxt, nxt + 1
        return acc

    var = 2 * k  # leaf of variable 0
    left = chain([t for i in range(k) for t in (i, var + i)] + [var + k + v for v in range(fa)])
    right = chain([k + i for i in range(k)] + [var + k + fa + v for v in range(fb)])
    chain([left, right])

    def exact(q):
        J = np.arange(1 << (fa + fb), dtype=np.uint64)
        z = np.ones_like(J)
        for i in range(k):
            def side(s):
                vs, t = sides[s][1:], np.array([x % q for x in tables[s]], dtype=np.uint64)
                at = sum((((J >> np.uint64(v - k)) & np.uint64(1)) << np.uint64(1 + j) for j, v in enumerate(vs)), np.uint64(0))
                return t[at], t[at + np.uint64(1)]
            (t0, t1), (u0, u1) = side(i), side(k + i)
            z = z * ((t0 * u0 % np.uint64(q) + t1 * u1 % np.uint64(q)) % np.uint64(q)) % np.uint64(q)
        return z

    return f, order, exact


@pytest.mark.parametrize("R,wide", [(1, False), (2, False), (2, True), (4, False), (4, True)])
@pytest.mark.parametrize("fa,fb,k,kernel", [
    (9, 7, 11, "block_32x16"), (8, 8, 8, "block_32x16"), (5, 11, 11, "block_32x16"),
    (9, 8, 9, "block_32x32"), (9, 9, 9, "block_32x32"), (5, 12, 12, "block_32x32"),
    (10, 9, 10, "block_64x32"), (6, 13, 13, "block_64x32"), (12, 8, 4, "block_64x32"),
    (9, 9, 3, "tile"), (11, 9, 2, "tile"), (8, 8, 3, "step"), (12, 4, 5, "block_32x16"), (13, 3, 6, "step"), (13, 4, 2, "outer"),
])
def test_kernel_of_a_step(fa, fb, k, kernel, R, wide):
    f, order, exact = _formula(fa, fb, k, 100 * fa + 10 * fb + k)
    p = tnc.plan(tnc.build_network(f), order=order, n_open=fa + fb)
    small = tnc.plan_formula(I.worked_example(), heuristic="gn")  # (a group: nothing in one launch)
    r = tnc.contract_many([p, small], n_residues=R, primes=WIDE[:R] if wide else None)[0]
    ran = tnc.last_kernel_launches()
    assert ran[kernel] >= 1, ran  # (the two sides have steps of their own with one small operand)
    for name in ("block_64x32", "block_32x32", "block_32x16", "tile"):
        assert ran[name] == (1 if name == kernel else 0), (name, ran)
    assert ran["total"] == sum(v for n, v in ran.items() if n != "total")
    assert np.array_equal(r.residues, np.stack([exact(q) for q in r.primes], axis=1))


@pytest.mark.parametrize("R,launches", [(1, 1), (4, 1), (8, 2), (3, 1)])
def test_small_formula_is_one_launch(R, launches):
    """(More than one residue group: the CRT is a launch of its own.)"""
    f = I.cubic_vertex_cover(70, 0)
    p = tnc.plan_formula(f, heuristic="greedy", rank_cap=28)
    assert tnc.contract(p, n_residues=R).residues.tolist() == oracle.residues(oracle.count(f, max_rank=28), tnc.default_primes(R))
    ran = tnc.last_kernel_launches()
    assert ran["one_launch"] == 1 and ran["crt_warp"] == launches - 1 and ran["total"] == launches


def test_kernels_of_the_other_paths():
    f = I.cubic_vertex_cover(100, 2)  # a dot product over 2^20 shared values at the end
    p = tnc.plan_formula(f, heuristic="bisect", rank_cap=24)
    want = oracle.count(f, max_rank=24)
    for path, R, kernels in (("int64", 4, ("splitk_partial", "splitk_final", "level", "leaf_fill", "extract")),
                             ("tc", 4, ("rns_pack", "p8_gemm", "rns_join", "splitk_partial")),
                             ("tc_p8", 12, ("p8_pack", "p8_gemm", "splitk_partial"))):
        assert tnc.contract(p, n_residues=R, path=path).residues.tolist() == oracle.residues(want, tnc.default_primes(R, path))
        ran = tnc.last_kernel_launches()
        assert all(ran[k] >= 1 for k in kernels), (path, ran)
        assert ran["one_launch"] == 0 and ran["total"] == sum(v for n, v in ran.items() if n != "total")
        assert path == "tc" or ran["rns_pack"] == 0
