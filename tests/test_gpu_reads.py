"""Reads of a 3D lattice that steps on moments take their values from its next
step, made for the first of them: they see the body force, the state and the
solid of the moment of the read, leave the trajectory alone, and hold what a
lattice in the two-pass form (which forms them node by node) gives: FP64 to 1e-12
of each field's scale, velocities (cancelling sums) to 5e-12 of the speed.
"""
import pytest

import synthetic as S
from dsm_helpers import gpu_lattice, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_19941_gb300 import _lib  # noqa: E402

FIELDS = ("C2", "C3", "mu", "ux", "uy", "uz", "pt", "rho", "tau")


def _case(shape=(45, 13, 9)):
    sd = S.pillars_sd(shape, 2, 6, 16, 4, offset=3)
    c2 = S.layer_c2(shape, 2, 3, 7, 1.0, sd, 1.0).ravel() + S.perturbation(3, sd.size)
    return S.Case("reads", "D3Q19", shape, sd.ravel(), c2, theta_deg=110.0, g23=0.01, g12=0.01,
                  alpha_s=1.0, body=(2e-6, -1e-6, -5e-6))


def test_fields_and_observables_equal_the_two_pass_forms():
    one, two = gpu_lattice(_case(), "f64"), gpu_lattice(_case(), "f64")
    two.set_step_form("two_pass")
    one.step(6)
    two.step(6)
    oa, ob = one.observables(), two.observables()
    for k in FIELDS:
        a, b = one.field(k).cpu().numpy(), two.field(k).cpu().numpy()
        if k[0] == "u":
            assert abs(a - b).max() < 5e-12 * ob["max_u"], k
        else:
            assert rel_err(a, b) < 1e-12, k
    for k, tol in (("mass_c2", 1e-12), ("mass_c1", 1e-12), ("kinetic", 1e-11), ("max_u", 5e-12)):
        assert abs(oa[k] - ob[k]) <= tol * abs(ob[k]), k


@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_reads_see_the_present_force_and_state(prec):
    a, b = gpu_lattice(_case(), prec), gpu_lattice(_case(), prec)
    a.step(5)
    a.field("uz")
    a.set_body_force((0.0, 0.0, 3e-5))
    b.step(5)
    b.set_body_force((0.0, 0.0, 3e-5))
    assert torch.equal(a.field("uz"), b.field("uz"))
    a.observables()
    a.step(4)
    b.step(4)
    a.field("pt")
    for lat in (a, b):
        nb = _lib.dsm_batch_scratch_bytes([lat.h])
        _lib.dsm_batch_step([lat.h], [3], torch.empty(nb, dtype=torch.uint8, device="cuda"), nb)
    assert torch.equal(a.field("mu"), b.field("mu"))
    a.set_fluid(b.field("C2"))
    b.set_fluid(b.field("C2"))
    assert torch.equal(a.field("mu"), b.field("mu"))
    a.step(2)
    b.step(2)
    assert all(torch.equal(u, v) for u, v in zip(a.populations(), b.populations()))
