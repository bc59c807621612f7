"""GPU tests of the halves that the digit stencil computes in the kind's own arithmetic
because one scale per column will not do: the values are the CUDA-core kernel's, and the
time is close to that kernel's."""
import json

import numpy as np
import pytest

import hisq_inputs as hi
from oracle import hisq
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

FX = 8192 + 1
CORES = {"f64": 512 + 2, "f64_native": 1}


def flag(psi, prec):
    """psi made a block that one scale per column does not hold: an entry of 1e33
    (double-float), a site a factor of 1e6 below its column (native FP64)."""
    if prec == "f64":
        psi[len(psi) // 2, 7, 2] = 1e33
    else:
        psi[:, 7] *= 1e-6
    return psi


def column_err(a, b):
    return max(gh.rel_err(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("prec", list(CORES))
@pytest.mark.parametrize("dims,N", [((2, 4, 6, 2), 2), ((4, 6, 4, 8), 5), ((6, 4, 4, 10), 16),
                                    ((4, 4, 4, 4), 33), ((16, 16, 16, 8), 16), ((16, 16, 16, 16), 15)])
def test_values_are_the_cuda_core_kernels(prec, dims, N):
    """Either half alone and the operator, then blocks that one scale does hold on the same
    handle (the flag does not outlive its call).  On the two larger lattices a thread takes
    two and four right-hand sides, a ragged number of them in the last."""
    psi = flag(hi.gaussian_sources(dims, N, seed=31), prec)
    good = hi.gaussian_sources(dims, N, seed=32)
    outs = []
    for v in (FX, CORES[prec]):
        s, _, _ = gh.make_solver(dims, 0.1, prec=prec, seed=33, max_rhs=N, dslash_variant=v)
        outs.append([gh.to_np(o) for o in (s.dslash(psi, 0), s.dslash(psi, 1), s.apply_MdagM(psi),
                                           s.dslash(good, 1), s.apply_MdagM(good))])
    for i in range(5):
        assert column_err(outs[0][i], outs[1][i]) < gh.TOL[prec], i


@pytest.mark.parametrize("prec", list(CORES))
def test_time_is_close_to_the_cuda_core_kernels(prec):
    """Within a quarter of the CUDA-core kernel chosen outright (4 and 1 % when measured;
    one right-hand side a thread took 1.5 times as long in double-float)."""
    torch = gh.torch_mod()
    dims, N, V = (32, 32, 32, 32), 16, 32 ** 4
    gen = torch.Generator(device="cuda").manual_seed(34)
    links = 0.3 * torch.randn((2, 4, V, 3, 3), dtype=torch.complex128, device="cuda", generator=gen)
    psi = flag(torch.randn((N, V // 2, 3), dtype=torch.complex128, device="cuda", generator=gen), prec)
    ms = []
    for v in (FX, CORES[prec]):
        s, _, _ = gh.make_solver(dims, 0.1, prec=prec, links=links, max_rhs=N, dslash_variant=v)
        best = 1e30
        for rep in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(3):
                s.apply_MdagM(psi)
            b.record()
            b.synchronize()
            if rep:
                best = min(best, a.elapsed_time(b))
        ms.append(best)
    assert ms[0] <= 1.25 * ms[1], ms


@pytest.mark.parametrize("decades", [0.02, 0.25, 2.0])
@pytest.mark.parametrize("N", [2, 8, 11, 16, 17, 40])
def test_falling_columns_in_double_float(N, decades):
    """A column that falls from time slice to time slice (0.3, 4 and 30 decades over the
    lattice) keeps double-float's accuracy in every slice, as an operator and as a half."""
    dims, mass = (4, 4, 4, 16), 0.1
    psi = hi.gaussian_sources(dims, N, seed=36)
    t = (np.arange(psi.shape[1]) * 2) // (4 * 4 * 4)
    psi *= (10.0 ** (-decades * t))[None, :, None]
    s, fat, lng = gh.make_solver(dims, mass, seed=37, max_rhs=N, dslash_variant=FX)
    for out, ref in ((s.dslash(psi, 1), hisq.dslash(dims, fat, lng, psi, 1)),
                     (s.apply_MdagM(psi), hisq.apply_A(dims, fat, lng, mass, psi))):
        out = gh.to_np(out)
        for k in range(dims[3]):
            assert gh.rel_err(out[:, t == k], ref[:, t == k]) < gh.TOL["f64"], k


@pytest.mark.parametrize("prec", list(CORES))
@pytest.mark.parametrize("small", [2.0 ** -4, 2.0 ** -30])
def test_links_of_very_different_size(prec, small):
    """Long links far below the fat ones, on a block that is zero but in one time slice: the
    slices that only the long links reach are as exact as the others."""
    dims, N = (4, 4, 4, 16), 5
    fat, lng = hi.random_links(dims, 38)
    lng = lng * small
    psi = hi.gaussian_sources(dims, N, seed=39)
    t = (np.arange(psi.shape[1]) * 2) // (4 * 4 * 4)
    psi[:, t != 5] = 0
    s, _, _ = gh.make_solver(dims, 0.1, prec=prec, links=(fat, lng), max_rhs=N, dslash_variant=FX)
    out, ref = gh.to_np(s.dslash(psi, 1)), hisq.dslash(dims, fat, lng, psi, 1)
    for k in range(dims[3]):
        if not np.any(ref[:, t == k]):
            assert not np.any(out[:, t == k]), k
        else:
            assert gh.rel_err(out[:, t == k], ref[:, t == k]) < gh.TOL[prec], k


@pytest.mark.parametrize("N", [3, 8, 16, 24])
@pytest.mark.parametrize("tracked", [False, True])
def test_point_sources_in_a_solve(tmp_path, N, tracked):
    """The first iterations of a solve from point sources run flagged halves, the later ones
    digits, with the maxima of P found by the stencil or left by the tensor-core update: the
    iterations of the cp.async kernel (one more or less), and tol on the oracle's residual."""
    torch = gh.torch_mod()
    dims, mass, tol = (8, 8, 8, 12), 0.1, 1e-11
    vh = int(np.prod(dims)) // 2
    b = np.zeros((N, vh, 3), dtype=np.complex128)
    for j in range(N):
        b[j, (vh // 2 + 37 * j) % vh, j % 3] = 1
    dev = torch.cuda.get_device_name().replace(" ", "_")
    iters = []
    for v in (CORES["f64"], FX):
        path = tmp_path / f"{v}.json"
        flags = 8 | (8 << 8) | (8 << 16) | ((1 << 24) if tracked else 0)
        path.write_text(json.dumps({f"blas/8.8.8.12/kind0/N{N}/{dev}": flags}))
        s, fat, lng = gh.make_solver(dims, mass, seed=39, max_rhs=N, dslash_variant=v)
        s.set_tune_cache(path)
        X, info = s.solve(b, tol=tol)
        assert info["status"] == 0
        r = (b - hisq.apply_A(dims, fat, lng, mass, gh.to_np(X))).reshape(N, -1)
        assert np.linalg.norm(r, axis=1).max() <= tol * 1.01
        iters.append(info["iters"])
    assert abs(iters[0] - iters[1]) <= 1, iters
