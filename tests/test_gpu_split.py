"""GPU tests of the hop-split stencil (4 or 16 lanes per output) and of the layout
conversions at the edges of their tiles (32 sites, 16 columns)."""
import json

import numpy as np
import pytest

import hisq_inputs as hi
from oracle import hisq
from tests import gpu_helpers as gh

pytestmark = pytest.mark.gpu

KIND = {"f64": 0, "mixed_f32": 1, "f64_native": 2}
SPLIT = 65536


@pytest.mark.parametrize("prec", list(KIND))
@pytest.mark.parametrize("lanes", [4, 16])
@pytest.mark.parametrize("dims,N,anti", [((2, 2, 2, 2), 1, False), ((4, 6, 2, 4), 3, True),
                                         ((4, 4, 6, 8), 9, False), ((6, 2, 4, 4), 64, True)])
def test_hop_split(tmp_path, prec, lanes, dims, N, anti):
    """The kernel forced through the tuning cache, against the oracle."""
    torch = gh.torch_mod()
    name = torch.cuda.get_device_name().replace(" ", "_")
    key = f"stencil/{'.'.join(map(str, dims))}/kind{KIND[prec]}/N{N}/recon0/{name}"
    path = tmp_path / "tune.json"
    path.write_text(json.dumps({key: SPLIT + lanes}, indent=1) + "\n")
    s, fat, lng = gh.make_solver(dims, 0.1, prec=prec, seed=81, max_rhs=N, antiperiodic_t=anti)
    s.set_tune_cache(path)
    psi = hi.gaussian_sources(dims, N, seed=82 + N)
    for p in (0, 1):
        ref = hisq.dslash(dims, fat, lng, psi, p, antiperiodic_t=anti)
        assert gh.rel_err(gh.to_np(s.dslash(psi, p)), ref) < gh.TOL[prec]
    ref = hisq.apply_A(dims, fat, lng, 0.1, psi, antiperiodic_t=anti)
    assert gh.rel_err(gh.to_np(s.apply_MdagM(psi)), ref) < gh.TOL[prec]
    assert json.loads(path.read_text())[key] == SPLIT + lanes  # not timed again


@pytest.mark.parametrize("dims,N", [((2, 2, 2, 2), 1), ((4, 4, 4, 2), 15), ((4, 4, 4, 2), 16),
                                    ((6, 2, 4, 6), 17), ((2, 6, 6, 4), 33), ((4, 6, 2, 4), 64)])
def test_layout_round_trip(dims, N):
    """Y + X 0 through the internal layout and back: every value once, in place
    (double-float holds 48 bits)."""
    s, _, _ = gh.make_solver(dims, 0.1, seed=83, max_rhs=N)
    vh = int(np.prod(dims)) // 2
    y = (np.arange(N * vh * 3, dtype=np.float64) + 0.25j).reshape(N, vh, 3)
    out = gh.to_np(s.block_caxpy(hi.gaussian_sources(dims, N, 84), np.zeros((N, N)), y))
    assert np.array_equal(out, y)
