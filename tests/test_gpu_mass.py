"""FP32 lattices on moments conserve their liquid: C + d is rounded without bias.

The bound: each rounding errs by at most a unit of C's last place u = 2^-24 (C
below 1), with a standard deviation of at most u / 2; n nodes and s steps that err
independently give u / 2 sqrt(n s).  Six standard deviations, doubled for nodes
that round alike by symmetry, over the mass.
"""
import math

import pytest

import synthetic as S
from dsm_helpers import gpu_lattice

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2504_19941_gb300 as P  # noqa: E402


def _case(shape, radius):
    sd = S.slab_sd(shape, len(shape) - 1, 0, 4)
    centre = [s / 2 for s in shape]
    centre[-1] = 10.0
    c2 = S.drop_c2(shape, centre, radius, 1.0, sd, 1.0).ravel() + S.perturbation(3, sd.size)
    return S.Case("mass", "D2Q9" if len(shape) == 2 else "D3Q19", shape, sd.ravel(), c2,
                  theta_deg=100.0, g23=2.5e-3, g12=2.5e-3, alpha_s=1.0)


def _bound(n, steps, mass):
    return 12.0 * 2.0 ** -25 * math.sqrt(n * steps) / mass


@pytest.mark.parametrize("shape,radius,steps,form", [
    ((24, 24, 24), 8.0, 5000, "auto"), ((24, 24, 24), 8.0, 5000, "two_pass"),
    ((64, 48, 40), 12.0, 4000, "auto"), ((96, 64), 16.0, 20000, "auto")])
@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_liquid_is_conserved(shape, radius, steps, form, prec):
    if prec == "f16" and (len(shape) == 2 or shape[0] < 32):
        pytest.skip("16-bit lattices of this size keep their populations")
    lat = gpu_lattice(_case(shape, radius), prec)
    lat.set_step_form(form)
    m0 = lat.observables()["mass_c2"]
    lat.step(steps)
    drift = lat.observables()["mass_c2"] / m0 - 1.0
    assert abs(drift) < _bound(lat.n, steps, m0), drift


def test_each_of_three_fluids_is_conserved():
    shape, steps = (32, 24, 24), 20000
    case = _case(shape, 8.0)
    n = math.prod(shape)
    p = P.make_params("D3Q19", shape, "f32", theta_deg=90.0, alpha_s=1.0)
    ml = P.MultiLattice(p, 3, (7.5e-3,) * 4, (1.0,) * 3, (1.0,) * 3)
    ml.set_solid_distance(torch.as_tensor(case.solid_sd, dtype=torch.float32, device="cuda"))
    c2 = torch.as_tensor(case.c2, dtype=torch.float32, device="cuda")
    left = (torch.arange(n, device="cuda") % shape[0] < shape[0] // 2).float()
    ml.set_fluids(torch.stack([c2 * left, c2 * (1 - left)]).contiguous())
    m0 = [float(ml.field("C", f).double().sum()) for f in range(2)]
    ml.step(steps)
    for f in range(2):
        drift = float(ml.field("C", f).double().sum()) / m0[f] - 1.0
        assert abs(drift) < _bound(n, steps, m0[f]), (f, drift)
