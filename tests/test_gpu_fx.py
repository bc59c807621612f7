"""GPU tests of the digit stencil (exact 8-bit digit products on the tensor cores;
double-float and native FP64) at the edges of its range: widths around its row
blocks of 8 and 16, extents of 2, both parities, antiperiodic time, and the blocks
one scale per column cannot represent, which take the kind's own arithmetic."""
import numpy as np
import pytest

import hisq_inputs as hi
from oracle import hisq
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

FX = 8192 + 1
PLAIN = {"f64": 512 + 2, "f64_native": 1}


@pytest.mark.parametrize("prec", ["f64", "f64_native"])
@pytest.mark.parametrize("dims,N,anti", [
    ((4, 4, 4, 4), 2, False), ((2, 4, 6, 2), 7, True), ((6, 2, 4, 8), 8, False),
    ((4, 6, 2, 10), 9, True), ((6, 8, 4, 6), 17, False), ((4, 4, 6, 8), 33, True),
    ((6, 4, 4, 4), 64, False)])
def test_widths_and_extents(prec, dims, N, anti):
    s, fat, lng = gh.make_solver(dims, 0.1, prec=prec, seed=71, max_rhs=N, dslash_variant=FX,
                                 antiperiodic_t=anti)
    psi = hi.gaussian_sources(dims, N, seed=72 + N)
    for p in (0, 1):
        ref = hisq.dslash(dims, fat, lng, psi, p, antiperiodic_t=anti)
        assert gh.rel_err(gh.to_np(s.dslash(psi, p)), ref) < gh.TOL[prec]
    ref = hisq.apply_A(dims, fat, lng, 0.1, psi, antiperiodic_t=anti)
    assert gh.rel_err(gh.to_np(s.apply_MdagM(psi)), ref) < gh.TOL[prec]


@pytest.mark.parametrize("prec", ["f64", "f64_native"])
@pytest.mark.parametrize("N", [3, 16])
@pytest.mark.parametrize("value", [np.nan, np.inf, 1e35])
def test_unscalable_columns(prec, N, value):
    """A NaN, an infinity or a huge entry: the same finite and non-finite entries
    as the CUDA-core kernel, and the same finite values."""
    dims = (4, 6, 4, 8)
    psi = hi.gaussian_sources(dims, N, seed=75)
    psi[1, 7, 2] = value
    out = []
    for v in (FX, PLAIN[prec]):
        s, _, _ = gh.make_solver(dims, 0.1, prec=prec, seed=73, max_rhs=N, dslash_variant=v)
        out.append(gh.to_np(s.apply_MdagM(psi)))
    a, b = out
    assert np.array_equal(np.isfinite(a), np.isfinite(b))
    f = np.isfinite(a)
    scale = np.abs(np.where(f, b, 0)).max(axis=(1, 2), keepdims=True)
    assert np.all(np.abs(a - b)[f] <= (gh.TOL[prec] * np.broadcast_to(scale, a.shape))[f])


def test_wide_range_within_a_column_native():
    """Native FP64 resolves every site of a column to 53 bits of itself, however
    far it lies below the column's maximum (a smeared point source)."""
    dims = (4, 4, 4, 16)
    N = 4
    psi = hi.gaussian_sources(dims, N, seed=76)
    t = (np.arange(psi.shape[1]) * 2) // (4 * 4 * 4)
    psi *= (10.0 ** (-2.0 * t))[None, :, None]
    s, fat, lng = gh.make_solver(dims, 0.1, prec="f64_native", seed=74, max_rhs=N, dslash_variant=FX)
    out = gh.to_np(s.dslash(psi, 1))
    ref = hisq.dslash(dims, fat, lng, psi, 1)
    for k in range(dims[3]):
        sl = t == k
        assert gh.rel_err(out[:, sl], ref[:, sl]) < gh.TOL["f64_native"], k


def test_zero_columns_and_zero_links():
    dims = (4, 4, 4, 6)
    N = 5
    for prec in ("f64", "f64_native"):
        fat, lng = hi.random_links(dims, 77)
        s, _, _ = gh.make_solver(dims, 0.1, prec=prec, links=(fat, 0 * lng), max_rhs=N, dslash_variant=FX)
        psi = hi.gaussian_sources(dims, N, seed=78)
        psi[2] = 0
        out = gh.to_np(s.dslash(psi, 0))
        assert np.all(out[2] == 0)
        assert gh.rel_err(out, hisq.dslash(dims, fat, 0 * lng, psi, 0)) < gh.TOL[prec]
        s, _, _ = gh.make_solver(dims, 0.1, prec=prec, links=(0 * fat, 0 * lng), max_rhs=N, dslash_variant=FX)
        assert np.all(gh.to_np(s.dslash(psi, 0)) == 0)
