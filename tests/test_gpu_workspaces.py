"""The same counts in every workspace that a call takes, from what it asks for down
to the least: residue groups side by side, one at a time, one residue at a time,
and TNC_PATH_TC without room for its operand planes (CUDA cores alone)."""
import numpy as np
import pytest

import oracle
from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc
from test_gpu_dense_shapes import WIDE, _formula

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()


def _sizes(plans, path, R, sliced, asked):
    out = [asked]
    while out[-1]:
        out.append(tnc.workspace_bytes_below(plans, R, out[-1], path, sliced=sliced))
    return out[:-1]


@pytest.mark.parametrize("path,R", [("int64", 7), ("tc", 1), ("tc", 3), ("tc", 4), ("tc", 7), ("tc_p8", 3), ("tc_p8", 7), ("tc_p8", 13)])
def test_counts_in_every_workspace(path, R):
    import torch
    f = I.cubic_vertex_cover(90, 4)
    p = tnc.plan_formula(f, heuristic="bisect", rank_cap=24)
    want = oracle.residues(oracle.count(f, max_rank=24), tnc.default_primes(R, path))
    small = tnc.plan_formula(I.cubic_vertex_cover(70, 0), heuristic="greedy", rank_cap=28)
    dense = "p8_gemm" if path == "tc_p8" else "tc_gemm"
    ran = []
    for size in _sizes([p], path, R, False, tnc.workspace_bytes(p, R, path)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        assert tnc.contract(p, R, path=path, workspace=ws).residues.tolist() == want, size
        ran.append(tnc.last_launch_counts()[dense] > 0)
        many = tnc.contract_many([p, small, p], R, path=path, workspace=ws)
        assert many[0].residues.tolist() == many[2].residues.tolist() == want, size
    if path == "tc" and R > 1:  # (one residue at a time leaves room for planes beside a smaller arena)
        assert ran.count(True) >= 2
    if path != "int64":
        assert ran[0] and (path == "tc_p8") <= ran[-1]
    assert len(ran) >= (1 if path == "int64" else 2)
    # the last choice of TNC_PATH_TC: what TNC_PATH_INT64 has at least
    ws = torch.empty(_sizes([p], "int64", R, False, tnc.workspace_bytes(p, R))[-1], dtype=torch.uint8, device="cuda")
    if path == "tc":
        assert tnc.contract(p, R, path=path, workspace=ws).residues.tolist() == want


@pytest.mark.parametrize("R,wide", [(1, False), (3, True), (4, False)])
@pytest.mark.parametrize("fa,fb,k", [(9, 7, 11), (7, 5, 13), (8, 6, 8), (7, 6, 16), (10, 9, 10)])
def test_dense_steps_in_what_the_workspace_leaves(fa, fb, k, R, wide):
    """TNC_PATH_TC between its smallest size of its own and what TNC_PATH_INT64 takes: one
    residue at a time, a step's shared values in parts that are added (more joins than steps)."""
    import torch
    f, order, exact = _formula(fa, fb, k, 100 * fa + 10 * fb + k)
    p = tnc.plan(tnc.build_network(f), order=order, n_open=fa + fb)
    primes = WIDE[:R] if wide else None
    want = tnc.contract(p, R, primes=primes, path="tc")
    assert np.array_equal(want.residues, np.stack([exact(q) for q in want.primes], axis=1))
    own, least = _sizes([p], "tc", R, False, tnc.workspace_bytes(p, R, "tc"))[-2:]
    if least < _sizes([p], "int64", R, False, tnc.workspace_bytes(p, R))[-1]:
        return  # one residue at a time takes less than all of them on the CUDA cores: nothing in between
    parts = 0
    for i in range(13):
        size = least + (own - least) * i // 13 // 256 * 256
        r = tnc.contract(p, R, primes=primes, path="tc", workspace=torch.empty(size, dtype=torch.uint8, device="cuda"))
        parts += tnc.last_kernel_launches()["rns_join"] > tnc.last_launch_counts()["tc_gemm"]
        assert r.residues.tolist() == want.residues.tolist(), size
    assert parts >= 1
    with pytest.raises(ValueError):
        tnc.contract(p, R, primes=primes, path="tc", workspace=torch.empty(least - 256, dtype=torch.uint8, device="cuda"))


@pytest.mark.parametrize("path,R", [("int64", 5), ("tc", 3), ("tc_p8", 6)])
def test_slices_in_every_workspace(path, R):
    import torch
    f = I.cubic_vertex_cover(90, 4)
    plans, _ = tnc.plan_sliced(f, 2, heuristic="bisect", rank_cap=24)
    want = oracle.residues(oracle.count(f, max_rank=24), tnc.default_primes(R, path))
    asked = tnc.workspace_bytes_many(plans, R, path, group=len(plans)) + 65536
    sizes = _sizes(plans, path, R, True, asked)
    assert len(sizes) >= 2
    for size in sizes:
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        assert tnc.contract_sliced(plans, R, path=path, workspace=ws).residues.tolist() == want, size
    with pytest.raises(ValueError):
        tnc.contract_sliced(plans, R, path=path, workspace=torch.empty(sizes[-1] - 256, dtype=torch.uint8, device="cuda"))
