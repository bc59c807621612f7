"""GPU tests of the tensor-core block BLAS of the double-float and FP32 kinds (update,
W update, Gram) at widths around its paddings of 8, 16 and 32 columns, through whole
solves with each kernel forced by the tuning cache."""
import json

import numpy as np
import pytest

import hisq_inputs as hi
from oracle import hisq
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

KIND = {"f64": 0, "mixed_f32": 1}
UPD, WGRAM, GRAM = 1 << 24, 1 << 25, 1 << 26


@pytest.mark.parametrize("prec", list(KIND))
@pytest.mark.parametrize("N", [3, 8, 9, 15, 17, 31, 32])
def test_forced_kernels_converge(tmp_path, prec, N):
    """Each kernel alone and all together meet tol on the oracle's residual in as many
    iterations as the CUDA-core kernels (one more or less for double-float, a tenth for
    FP32); 6 x 4 x 6 x 10 has 2160 rows, a whole number of 16-row tiles, 33 and 3/4
    tiles of 64."""
    torch = gh.torch_mod()
    dims, mass, tol = (6, 4, 6, 10), 0.1, 1e-11
    dev = torch.cuda.get_device_name().replace(" ", "_")
    b = hi.gaussian_sources(dims, N, seed=91 + N)
    iters = {}
    for name, flags in (("cores", 0), ("upd", UPD), ("wgram", WGRAM), ("gram", GRAM),
                        ("all", UPD | WGRAM | GRAM)):
        path = tmp_path / f"{name}.json"
        path.write_text(json.dumps({f"blas/6.4.6.10/kind{KIND[prec]}/N{N}/{dev}":
                                    8 | (8 << 8) | (8 << 16) | flags}))
        s, fat, lng = gh.make_solver(dims, mass, prec=prec, seed=90, max_rhs=N)
        s.set_tune_cache(path)
        X, info = s.solve(b, tol=tol)
        assert info["status"] == 0, name
        X = gh.to_np(X)
        r = (b - hisq.apply_A(dims, fat, lng, mass, X)).reshape(N, -1)
        rel = np.linalg.norm(r, axis=1) / np.linalg.norm(b.reshape(N, -1), axis=1)
        assert rel.max() <= tol * 1.01, (name, rel)
        iters[name] = info["iters"]
    for name in iters:
        assert abs(iters[name] - iters["cores"]) <= (1 if prec == "f64" else iters["cores"] // 10), iters


@pytest.mark.parametrize("N", [3, 8, 16, 24])
def test_update_leaves_the_column_maxima(tmp_path, N):
    """The digit stencil scales P's columns by the maxima that the tensor-core update
    leaves: the solve takes the iterations that it takes when the stencil finds them
    itself (the CUDA-core update), through reliable updates, and meets tol."""
    torch = gh.torch_mod()
    dims, mass, tol = (6, 4, 6, 10), 0.1, 1e-11
    dev = torch.cuda.get_device_name().replace(" ", "_")
    b = hi.gaussian_sources(dims, N, seed=71 + N)
    iters = []
    for flags in (0, UPD):
        path = tmp_path / f"{flags}.json"
        path.write_text(json.dumps({f"blas/6.4.6.10/kind0/N{N}/{dev}":
                                    8 | (8 << 8) | (8 << 16) | flags}))
        s, fat, lng = gh.make_solver(dims, mass, seed=70, max_rhs=N, dslash_variant=8192 + 1)
        s.set_tune_cache(path)
        X, info = s.solve(b, tol=tol)
        assert info["status"] == 0 and info["reliable_updates"] >= 1
        r = (b - hisq.apply_A(dims, fat, lng, mass, gh.to_np(X))).reshape(N, -1)
        rel = np.linalg.norm(r, axis=1) / np.linalg.norm(b.reshape(N, -1), axis=1)
        assert rel.max() <= tol * 1.01, (flags, rel)
        iters.append(info["iters"])
    assert abs(iters[0] - iters[1]) <= 1, iters


@pytest.mark.parametrize("dims,N", [((16, 16, 16, 16), 8), ((16, 8, 12, 16), 14),
                                    ((16, 8, 12, 16), 17), ((12, 8, 8, 16), 31),
                                    ((12, 8, 8, 16), 32)])
def test_reliable_updates_of_the_fp32_iteration(dims, N):
    """Blocks large enough (V_h N^2 >= 2^21) that Q and P of a reliable update come from the
    tensor cores: the mixed solve meets tol on the oracle's residual, with at most twice the
    iterations of the double-float form, whose updates are the CUDA cores'."""
    mass, tol = 0.1, 1e-11
    b = hi.gaussian_sources(dims, N, seed=51 + N)
    iters = {}
    for prec in ("f64", "mixed_f32"):
        s, fat, lng = gh.make_solver(dims, mass, prec=prec, seed=50, max_rhs=N)
        X, info = s.solve(b, tol=tol)
        assert info["status"] == 0 and info["reliable_updates"] >= 1
        r = (b - hisq.apply_A(dims, fat, lng, mass, gh.to_np(X))).reshape(N, -1)
        rel = np.linalg.norm(r, axis=1) / np.linalg.norm(b.reshape(N, -1), axis=1)
        assert rel.max() <= tol * 1.01, (prec, rel)
        iters[prec] = info["iters"]
    assert iters["mixed_f32"] <= 2 * iters["f64"], iters
