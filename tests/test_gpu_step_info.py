"""dsm_step_info and Lattice.single_pass say which form dsm_step runs, and a
given number of planes per block is taken: FP32 arithmetic with a density
contrast on both sides of the 180000 nodes from which the automatic form runs
two passes.  Which form ran shows in the end of the workspace: the padded copy of
C1, which only the one-pass step over populations writes.
"""
import pytest

import synthetic as S
from dsm_helpers import gpu_lattice, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_19941_gb300 import _lib  # noqa: E402


def _lattice(shape, prec, form="auto", zrun=0):
    sd = S.pillars_sd(shape, 4, 6, 16, 8, offset=3)
    c2 = S.layer_c2(shape, 2, 8, 20, 1.0, sd, 1.0).ravel() + S.perturbation(3, sd.size)
    case = S.Case("info", "D3Q19", shape, sd.ravel(), c2, theta_deg=110.0, g23=0.01, g12=0.01,
                  alpha_s=1.0)
    case.rho2, case.rho3, case.tau2, case.tau3 = 1.0, 0.2, 1.0, 0.7
    lat = gpu_lattice(case, prec)
    lat.set_step_form(form, zrun)
    return lat


@pytest.mark.parametrize("prec,shape,auto", [("f32", (56, 56, 57), True), ("f32", (64, 64, 45), False),
                                             ("f16", (64, 64, 45), False), ("f64", (64, 64, 45), True)])
def test_step_info_is_the_form_that_runs(prec, shape, auto):
    lat = _lattice(shape, prec)
    single, zrun = _lib.dsm_step_info(lat.h)
    assert lat.single_pass == bool(single) == auto
    assert (zrun > 0) == auto
    given, two = _lattice(shape, prec, "auto", 7), _lattice(shape, prec, "two_pass")
    assert _lib.dsm_step_info(given.h) == (1, 7) and _lib.dsm_step_info(two.h) == (0, 0)
    ran = []
    for x in (lat, given, two):
        x.workspace[-4 * x.n:].zero_()
        x.step(12)
        ran.append(bool(x.workspace[-4 * x.n:].any()))
    assert ran == [auto, True, False]
    fa, fg, ft = (x.populations()[0] for x in (lat, given, two))
    assert torch.equal(fa, fg if auto else ft)
    assert rel_err(fg.cpu().numpy(), ft.cpu().numpy()) < {"f64": 1e-13, "f32": 2e-6, "f16": 1e-3}[prec]
