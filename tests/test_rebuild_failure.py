"""A rebuild whose bounded wait ran out: every call that reads or maintains the values says so, and a
rebuild puts it right.  The failure is made on the host, by setting the word that such a rebuild
sets."""
import ctypes as C

import numpy as np
import pytest

import workloads as W
from tests import ctx_access


@pytest.fixture(scope="module")
def access(tmp_path_factory):
    return ctx_access.load(tmp_path_factory.mktemp("ctx_access"))


@pytest.fixture(scope="module")
def sta():
    from paper_2605_11673_gb300 import build
    build.build()
    import paper_2605_11673_gb300 as P
    P.load_library()
    return P


def test_every_reader_reports_it_before_any_device_work(sta, access):
    """On a context without device state (no GPU needed)."""
    L = sta.load_library()
    i32, i64, f64 = C.c_int32(), C.c_int64(), C.c_double()
    calls = {
        "apply_edits": lambda h: L.sta_apply_edits(h, None, 0, None),
        "apply_edits_noalloc": lambda h: L.sta_apply_edits_noalloc(h, None, 0, None),
        "last_touched": lambda h: L.sta_last_touched(h, C.byref(i64), None),
        "spmv": lambda h: L.sta_spmv(h, None, None, None, None),
        "solve": lambda h: L.sta_solve(h, None, None, None, 1e-8, 10, None, C.byref(i32), C.byref(f64), None),
        # rebuilds, as nothing has reported it yet
        "refold": lambda h: L.sta_refold(h, None),
        "full_rebuild": lambda h: L.sta_full_rebuild(h, None, 0, None),
        "set_policy": lambda h: L.sta_set_policy(h, 1, None),
    }
    for name, call in calls.items():
        h = access.ctx_new()
        access.ctx_set_fault(h, 1)
        assert call(h) == sta.STA_ECUDA, name
        assert b"earlier rebuild" in L.sta_last_error(), (name, L.sta_last_error())
        assert access.ctx_fault(h) == 1, name
        access.ctx_delete(h)


@pytest.mark.gpu
@pytest.mark.parametrize("again", ["refold", "full_rebuild", "set_policy"])
@pytest.mark.parametrize("graph", [False, True])
def test_a_rebuild_puts_it_right(sta, access, orc, again, graph):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if graph and again == "set_policy":
        pytest.skip("not allowed in graph mode")
    wl = W.plain_small(seed=3, frames=2)
    masks = wl.masks()
    P = orc.Pattern(wl.n_nodes, wl.tets)
    Ke, _ = orc.element_all(wl.X, wl.tets, wl.E, wl.nu)
    asm = sta.Assembler(wl.X, wl.tets, wl.E, wl.nu)
    asm.full_rebuild(wl.mask0)
    asm.dyn_setup(1000.0, 1e-3)
    if graph:
        asm.graph_enable(4096)
    x = torch.ones(asm.n_rows, dtype=torch.float64, device="cuda")
    free = torch.ones(asm.n_rows, dtype=torch.bool, device="cuda")
    rebuild = {"refold": asm.refold, "full_rebuild": lambda: asm.full_rebuild(masks[0]),
               "set_policy": lambda: asm.set_policy(sta.STA_POLICY_REFOLD)}[again]
    torch.cuda.synchronize()
    access.ctx_set_fault(asm.h, 1)
    reads = [lambda: asm.apply_edits(wl.frames[0]), lambda: sta.sta_apply_edits_noalloc(asm.h, wl.frames[0]),
             asm.last_touched, lambda: sta.sta_spmv(asm.h, x), lambda: sta.sta_solve(asm.h, x, free),
             asm.dyn_step, lambda: asm.dyn_apply(x)]
    for k, call in enumerate([rebuild] + reads):  # (a rebuild too, while nothing has reported it)
        with pytest.raises(sta.StaError) as e:
            call()
        assert e.value.status == sta.STA_ECUDA and "earlier rebuild" in str(e.value), k
    rebuild()
    asm.apply_edits(wl.frames[0])  # (refused before: the mask is still the first one)
    got = asm.values().cpu().numpy().view(np.uint64)
    assert np.array_equal(got, P.rebuild(Ke, masks[1]).view(np.uint64))
    assert asm.last_touched() > 0
    asm.close()
