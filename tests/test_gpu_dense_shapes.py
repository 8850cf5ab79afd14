"""One dense step of a chosen shape (2^fa rows, 2^fb columns, 2^k shared values)
with full-size residues, against exact integers.

The formula has k inner variables x_i, each in one weighted clause T_i(x_i,
a_(i mod fa)) and one U_i(x_i, b_(i mod fb)); the a and b are open.  The order
contracts the T side and the U side first, so the last step is the dense one;
its result is prod_i sum_x T_i(x, a) U_i(x, b), computed here modulo each prime
in integers: the tolerance is zero."""
import random

import numpy as np
import pytest

from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

pytestmark = pytest.mark.gpu

WIDE = [2147483647, 2147483629, 2147483587, 2147483579]


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


def _formula(fa, fb, k, seed):
    """(formula, order, exact entries); variables: x_0.., a_0.., b_0.."""
    rng = random.Random(seed)
    T = [[rng.getrandbits(32) for _ in range(4)] for _ in range(k)]
    U = [[rng.getrandbits(32) for _ in range(4)] for _ in range(k)]
    clauses = [(i, k + i % fa) for i in range(k)] + [(i, k + fa + i % fb) for i in range(k)]
    n_vars = k + fa + fb
    f = I.Formula(n_vars, clauses, [I.KIND_TABLE] * (2 * k), T + U, open_vars=list(range(k, n_vars)))
    nxt, order = 2 * k + n_vars, []

    def chain(ids):
        nonlocal nxt
        acc = ids[0]
        for j in ids[1:]:
            order.append((acc, j))
            acc, nxt = nxt, nxt + 1
        return acc

    var = 2 * k  # leaf of variable 0
    left = chain([chain([t for i in range(j, k, fa) for t in (i, var + i)] + [var + k + j]) for j in range(fa)])
    right = chain([chain([k + i for i in range(j, k, fb)] + [var + k + fa + j]) for j in range(fb)])
    chain([left, right])

    def exact(q):
        """The entries mod q (below 2^31: products of two residues fit 64 bits)."""
        J = np.arange(1 << (fa + fb), dtype=np.uint64)
        z = np.ones_like(J)
        for i in range(k):
            v = [sum(T[i][x + 2 * a] * U[i][x + 2 * b] for x in (0, 1)) % q for b in (0, 1) for a in (0, 1)]
            at = ((J >> np.uint64(i % fa)) & np.uint64(1)) + np.uint64(2) * ((J >> np.uint64(fa + i % fb)) & np.uint64(1))
            z = z * np.array(v, dtype=np.uint64)[at] % np.uint64(q)
        return z

    return f, order, exact


@pytest.mark.parametrize("path,R,wide", [("tc", 1, False), ("tc", 3, True), ("tc", 4, False), ("int64", 4, False),
                                         ("int64", 3, True), ("tc_p8", 5, False)])
@pytest.mark.parametrize("fa,fb,k", [(7, 5, 7), (5, 7, 9), (8, 6, 8), (9, 7, 11), (7, 6, 16), (4, 8, 8), (3, 10, 10), (9, 8, 9),
                                     (10, 9, 10), (5, 12, 12), (12, 8, 12)])
def test_dense_step(fa, fb, k, path, R, wide):
    f, order, exact = _formula(fa, fb, max(k, fa, fb), 100 * fa + 10 * fb + k)  # (every open variable has a clause)
    p = tnc.plan(tnc.build_network(f), order=order, n_open=fa + fb)
    r = tnc.contract(p, n_residues=R, primes=WIDE[:R] if wide else None, path=path)
    if path == "tc" and min(fa, fb) >= 5:
        assert tnc.last_launch_counts()["tc_gemm"] >= 1
    assert np.array_equal(r.residues, np.stack([exact(q) for q in r.primes], axis=1))
