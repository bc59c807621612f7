"""GPU tests of handles without the digit form of the links: where no call reads it, and where
memory is short."""
import ctypes as ct

import numpy as np
import pytest

import hisq_inputs as hi
from oracle import hisq
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 16)  # 8192 sites: all forms have the digit form


class Larger:
    """blockcg_workspace_bytes, the first answer as of a block that fills the device."""

    def __init__(self, lib, total):
        self.f, self.total = lib.blockcg_workspace_bytes, total

    def __call__(self, h, n):
        extra, self.total = self.total, 0
        return self.f(h, n) + extra


def out_of_memory_from(empty, limit):
    def f(*args, **kw):
        if args and args[0] == limit:
            raise gh.torch_mod().cuda.OutOfMemoryError("test")
        return empty(*args, **kw)
    return f


@pytest.mark.parametrize("short,prec,variant", [
    ("asked", "f64", 0), ("asked", "f64", 8192 + 1), ("asked", "f64_native", 0),
    ("asked", "f64_native", 8192 + 1), ("asked", "mixed_f32", 0), ("asked", "mixed_f16", 0),
    ("tried", "f64", 0), ("tried", "mixed_f32", 0)])
def test_short_of_memory(monkeypatch, short, prec, variant):
    """With no room for it the handle takes 2528 bytes a site less, and a smaller workspace;
    the operator and a solve meet the oracle (the tensor-core stencil asked for by name runs
    the cp.async or plain kernel)."""
    torch = gh.torch_mod()
    mass, N, tol = 0.1, 6, 1e-10
    links = hi.random_links(DIMS, 41)
    args = dict(prec=prec, links=links, max_rhs=N, dslash_variant=variant)
    full, _, _ = gh.make_solver(DIMS, mass, **args)
    if short == "asked":  # a large handle asks for the free memory
        total = torch.cuda.get_device_properties(0).total_memory
        monkeypatch.setattr(full.lib, "blockcg_workspace_bytes", Larger(full.lib, total))
        monkeypatch.setattr(torch.cuda, "mem_get_info", lambda device=None: (0, total))
    else:  # a small one tries
        monkeypatch.setattr(torch, "empty", out_of_memory_from(torch.empty, full.workspace.numel()))
    s, fat, lng = gh.make_solver(DIMS, mass, **args)
    monkeypatch.undo()
    V = int(np.prod(DIMS))
    assert 2528 * V <= full.gauge.numel() - s.gauge.numel() <= 2528 * V + 1024
    assert full.workspace.numel() - s.workspace.numel() == 384 * V // 2  # records of 8 columns
    b = hi.gaussian_sources(DIMS, N, seed=42) / np.sqrt(3 * V / 2)
    ref = hisq.apply_A(DIMS, fat, lng, mass, b)
    assert gh.rel_err(gh.to_np(s.apply_MdagM(b)), ref) < gh.TOL[prec]
    X, info = s.solve(b, tol=tol)
    assert info["status"] == 0
    r = (b - hisq.apply_A(DIMS, fat, lng, mass, gh.to_np(X))).reshape(N, -1)
    assert (np.linalg.norm(r, axis=1) / np.linalg.norm(b.reshape(N, -1), axis=1)).max() <= tol * 1.01
    # the storage may be exchanged: reloading the links keeps the handle as it is
    s.load_gauge(fat, lng)
    assert gh.rel_err(gh.to_np(s.apply_MdagM(b)), ref) < gh.TOL[prec]


def test_one_right_hand_side_and_limits():
    """A handle for single right-hand sides does without; less than the least is refused, and
    so is more than one right-hand side."""
    links = hi.random_links(DIMS, 43)
    s, fat, lng = gh.make_solver(DIMS, 0.1, links=links, max_rhs=1)
    least = s.lib.blockcg_gauge_bytes_min(s.h)
    assert s.gauge.numel() == least < s.lib.blockcg_gauge_bytes(s.h)
    b = hi.gaussian_sources(DIMS, 2, seed=44)
    ref = hisq.apply_A(DIMS, fat, lng, 0.1, b[:1])
    assert gh.rel_err(gh.to_np(s.apply_MdagM(b[:1])), ref) < gh.TOL["f64"]
    with pytest.raises(RuntimeError):
        s.apply_MdagM(b)
    f, l = s._dev(fat), s._dev(lng)
    assert s.lib.blockcg_load_gauge(s.h, ct.c_void_p(f.data_ptr()), ct.c_void_p(l.data_ptr()),
                                    ct.c_void_p(s.gauge.data_ptr()), least - 1) == 3
