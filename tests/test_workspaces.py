"""Which workspaces the contractions ask for and which they take, on the host (an
injected launch failure ends an accepted call before its first device call).
Counts in such workspaces: test_gpu_workspaces.py."""
import ctypes
import types

import pytest

from paper_1805_00475_gb300 import build as tnc_build
from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

PATHS = [("int64", 4), ("int64", 7), ("int64", 16), ("tc", 1), ("tc", 4), ("tc", 7), ("tc_p8", 1), ("tc_p8", 7), ("tc_p8", 20)]


@pytest.fixture(scope="module", autouse=True)
def built():
    tnc_build.build()
    yield
    tnc.inject_failure("none")


@pytest.fixture(scope="module")
def plans():
    return {n: tnc.plan_formula(I.cubic_vertex_cover(n, g), heuristic=h, rank_cap=32)
            for n, g, h in ((40, 0, "greedy"), (110, 6, "greedy"), (130, 3, "best"), (140, 0, "best"))}


def _accepted(p, path, R, size, call="tnc_contract"):
    o, _ = tnc._opts(R, None, path)
    c = tnc._count_buffers(1 << p.n_open, R)
    args = [ctypes.byref(o), ctypes.c_void_p(1 << 20), size, None, ctypes.byref(c[0])]
    arr = (ctypes.c_void_p * 1)(p.h.value)
    tnc.inject_failure("launch")
    rc = getattr(tnc.lib(), call)(*([p.h] if call == "tnc_contract" else [arr, 1]), *args)
    tnc.inject_failure("none")
    assert rc in (-3, -4)  # the injected failure, or too small
    return rc == -3


def _sizes(p, path, R):
    out = [tnc.workspace_bytes(p, R, path)]
    while out[-1]:
        out.append(tnc.workspace_bytes_below([p], R, out[-1], path))
        assert out[-1] < out[-2]
    return out[:-1]


@pytest.mark.parametrize("path,R", PATHS)
def test_sizes_that_work(plans, path, R):
    for p in plans.values():
        sizes = _sizes(p, path, R)
        assert all(_accepted(p, path, R, s) and _accepted(p, path, R, s, "tnc_contract_many") for s in sizes)
        assert not _accepted(p, path, R, sizes[-1] - 1) and not _accepted(p, path, R, sizes[-1] - 1, "tnc_contract_many")


def test_int64_asks_for_no_tensor_core_scratch(plans):
    for n, p in plans.items():
        assert len(_sizes(p, "int64", 4)) == 1  # one residue group: nothing but what it needs
        assert tnc.workspace_bytes(p, 4) <= tnc.lib().tnc_workspace_bytes(p.h, 4) >= tnc.workspace_bytes(p, 4, "tc")
        assert n < 130 or tnc.workspace_bytes(p, 4, "tc") > tnc.workspace_bytes(p, 4)


# what the library asked for when dense steps of TNC_PATH_TC took their operands
# from the arena and every residue group ran by itself
EARLIER = [
    (110, "int64", 4, 331182336), (110, "tc", 1, 89350912), (110, "tc", 4, 331182336), (110, "tc", 16, 331196672),
    (110, "tc_p8", 1, 83943936), (110, "tc_p8", 3, 159148544), (110, "tc_p8", 7, 317946112), (110, "tc_p8", 20, 317961728),
    (140, "int64", 4, 95417088), (140, "tc", 1, 24190208), (140, "tc", 4, 95417088), (140, "tc", 16, 95424256),
    (140, "tc_p8", 1, 14779904), (140, "tc_p8", 3, 29112320), (140, "tc_p8", 7, 57776896), (140, "tc_p8", 20, 57784576),
    (130, "int64", 4, 56147712), (130, "tc", 1, 20640256), (130, "tc", 4, 56147712), (130, "tc", 16, 56162048),
    (130, "tc_p8", 1, 15696640), (130, "tc_p8", 3, 22590208), (130, "tc_p8", 7, 36376576), (130, "tc_p8", 20, 36392192),
]


@pytest.mark.parametrize("n,path,R,size", EARLIER)
def test_earlier_workspaces_are_accepted(plans, n, path, R, size):
    assert _accepted(plans[n], path, R, size)


@pytest.mark.parametrize("R", [1, 3, 4, 16])
def test_tc_takes_what_int64_takes(plans, R):
    for p in plans.values():
        assert _accepted(p, "tc", R, _sizes(p, "int64", R)[-1])


@pytest.mark.parametrize("call", ["contract", "contract_many", "contract_sliced"])
def test_less_memory_on_the_device(plans, monkeypatch, call):
    """Without a workspace of the caller's, sizes that cannot be had are followed by smaller ones."""
    import torch
    p, tried, stream = plans[130], [], types.SimpleNamespace(cuda_stream=0)
    least = _sizes(p, "tc", 16)[-1] + 65536

    def empty(nbytes, dtype, device):
        tried.append(nbytes)
        if nbytes > limit:
            raise torch.cuda.OutOfMemoryError("no memory left")
        return types.SimpleNamespace(numel=lambda: nbytes, element_size=lambda: 1, data_ptr=lambda: 1 << 20)

    monkeypatch.setattr(torch, "empty", empty)
    run = {"contract": lambda: tnc.contract(p, 16, path="tc", stream=stream),
           "contract_many": lambda: tnc.contract_many([p, p], 16, path="tc", stream=stream)}
    if call == "contract_sliced":  # its sum is cleared before the first slice is looked at
        with pytest.raises(torch.cuda.OutOfMemoryError):
            limit = 1024
            tnc.contract_sliced([p, p], 16, path="tc", stream=stream)
        assert len(tried) >= 4 and tried == sorted(tried, reverse=True) and tried[-1] <= least
        return
    limit = least
    tnc.inject_failure("launch")
    with pytest.raises(tnc.TncError) as e:
        run[call]()
    assert e.value.code == -3 and len(tried) >= 3 and tried == sorted(tried, reverse=True) and tried[-1] <= least
    limit, tried = 1024, []
    with pytest.raises(torch.cuda.OutOfMemoryError):
        run[call]()
