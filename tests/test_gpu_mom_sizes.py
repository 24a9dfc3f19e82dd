"""The step on moments at the ends of what its rules give it: FP64 in 3D on both
sides of 32768 nodes and in 2D of 19456 and 77824, against the oracle to 1e-12;
FP32 on the smallest lattices, to the 1e-5 of the FP32 parity tests.
"""
import numpy as np
import pytest

import oracle as O
from dsm_helpers import compare, direction_map, gpu_fields, gpu_lattice, gpu_pops, oracle_params, \
    rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from test_gpu_mom import _case  # noqa: E402


@pytest.mark.parametrize("shape,prec,zrun", [
    ((33, 32, 32), "f64", 0), ((31, 40, 27), "f64", 5), ((66, 31, 17), "f64", 4),
    ((32, 32, 31), "f64", 0), ((152, 127), "f64", 0), ((152, 129), "f64", 0),
    ((304, 255), "f64", 0), ((304, 256), "f64", 0),
    ((1, 1, 1), "f32", 0), ((2, 3, 1), "f32", 0), ((31, 8, 3), "f32", 1), ((33, 9, 5), "f32", 2),
    ((3, 2), "f32", 0)])
def test_sizes_match_oracle(shape, prec, zrun):
    case = _case(shape)
    steps = 3
    lat = gpu_lattice(case, prec)
    lat.set_step_form("auto", zrun)
    lat.step(steps)
    kind = O.D2Q9 if case.lattice == "D2Q9" else O.D3Q19
    p = oracle_params(case, kind)
    c1 = O.solid_profile(case.solid_sd, case.alpha_s)
    f, g = O.lb_init(p, 2, c1, case.c2)
    f, g = O.lb_run(p, 2, c1, f, g, steps)
    errs = compare(gpu_fields(lat), O.lb_fields(p, 2, c1, f, g), ("C", "pt", "rho"))
    gf, gg = gpu_pops(lat, direction_map(kind))
    errs["f"], errs["g"] = rel_err(gf, f), rel_err(gg, g)
    assert max(errs.values()) < (1e-12 if prec == "f64" else 1e-5), errs
    assert np.isfinite(lat.observables()["max_u"])
