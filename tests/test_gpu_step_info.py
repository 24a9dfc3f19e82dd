"""dsm_step_info and Lattice.single_pass say which form dsm_step runs, and a
given number of planes per block is taken, also by large lattices with a density
contrast.  Which form ran shows in the end of the workspace: the padded copy of
C1, which only the one-pass step over populations writes.
"""
import pytest

import synthetic as S
from dsm_helpers import gpu_lattice, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2504_19941_gb300 as P  # noqa: E402
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


@pytest.mark.parametrize("prec,shape,zauto", [
    ("f32", (64, 64, 45), 2), ("f16", (64, 64, 45), 2), ("f64", (64, 64, 45), None),
    ("f32", (160, 160, 100), 12), ("f32", (160, 130, 101), 7)])
def test_step_info_is_the_form_that_runs(prec, shape, zauto):
    # (zauto: on 152 SMs; runs of more than 12 planes become runs of 7)
    lat = _lattice(shape, prec)
    single, zrun = _lib.dsm_step_info(lat.h)
    assert lat.single_pass and single == 1 and zrun > 0
    assert zauto is None or zrun == zauto
    given, two = _lattice(shape, prec, "auto", 7), _lattice(shape, prec, "two_pass")
    assert _lib.dsm_step_info(given.h) == (1, 7) and _lib.dsm_step_info(two.h) == (0, 0)
    ran = []
    for x in (lat, given, two):
        x.workspace[-4 * x.n:].zero_()
        x.step(12)
        ran.append(bool(x.workspace[-4 * x.n:].any()))
    assert ran == [True, True, False]
    fa, fg, ft = (x.populations()[0] for x in (lat, given, two))
    assert torch.equal(fa, fg)
    assert rel_err(fg.cpu().numpy(), ft.cpu().numpy()) < {"f64": 1e-13, "f32": 2e-6, "f16": 1e-3}[prec]


def _form(lat):
    """How the state is held: 1 f with g as g_eq, 2 moments, 3 f and quads."""
    return int(lat.state()[:32].view(torch.int32)[7])


def _plain(shape, prec, **kw):
    sd = S.slab_sd(shape, len(shape) - 1, 0, 1)
    case = S.Case("form", "D2Q9" if len(shape) == 2 else "D3Q19", shape, sd.ravel(),
                  0.5 + S.perturbation(3, sd.size), theta_deg=90.0, g23=0.01, g12=0.01, alpha_s=1.0)
    for k, v in kw.items():
        setattr(case, k, v)
    lat = gpu_lattice(case, prec)
    lat.step(2)
    return lat


@pytest.mark.parametrize("shape,zrun", [((32, 32, 32), 1), ((48, 48, 48), 2), ((64, 64, 64), 4),
                                        ((101, 101, 101), 10)])
def test_fp32_runs_of_planes_on_moments(shape, zrun):
    # on 152 SMs: one wave of blocks, fewer on each SM where that is faster
    assert _lib.dsm_step_info(_plain(shape, "f32").h) == (1, zrun)


@pytest.mark.parametrize("shape,form,zrun", [
    ((32, 32, 31), 1, None), ((32, 32, 32), 2, 1), ((33, 32, 33), 2, 2), ((40, 40, 40), 2, 3),
    ((64, 64, 64), 2, 8), ((24, 48, 48), 1, 0), ((31, 64, 64), 2, 0), ((128, 4, 100), 1, 0),
    ((300, 5, 100), 1, 0)])
def test_fp64_in_3d_steps_on_moments_where_that_is_faster(shape, form, zrun):
    # runs of planes: one block on each of 152 SMs, which share no FP64 pipe
    lat = _plain(shape, "f64")
    assert _form(lat) == form
    if zrun is not None:
        assert _lib.dsm_step_info(lat.h)[1] == zrun


@pytest.mark.parametrize("shape,contrast,form", [
    ((128, 120), False, 3), ((160, 120), False, 1), ((17, 1100), True, 1), ((256, 128), True, 1),
    ((512, 400), False, 1), ((512, 400), True, 3)])
def test_fp64_in_2d_steps_from_quads_where_that_is_faster(shape, contrast, form):
    kw = dict(tau3=0.6, **(dict(rho3=0.5) if contrast else {}))
    assert _form(_plain(shape, "f64", **kw)) == form
    assert _form(_plain(shape, "f32", **kw)) == 3


@pytest.mark.parametrize("shape,nfluid,prec,moments", [
    ((32, 32, 32), 4, "f64", False), ((40, 32, 40), 4, "f64", True), ((32, 32, 32), 3, "f64", True),
    ((32, 32, 32), 4, "f32", True)])
def test_four_fluids_in_fp64_step_on_moments_where_that_is_faster(shape, nfluid, prec, moments):
    # the workspace starts with f_0 of the rest state, 1/3, where populations are kept
    real = torch.float64 if prec == "f64" else torch.float32
    n = shape[0] * shape[1] * shape[2]
    p = P.make_params("D3Q19", shape, prec, theta_deg=90.0, alpha_s=1.0)
    ml = P.MultiLattice(p, nfluid, (0.02,) * (nfluid + 1), (1.0,) * nfluid, (1.0,) * nfluid)
    ml.set_solid_c1(torch.zeros(n, dtype=real, device="cuda"))
    ml.set_fluids(torch.full((nfluid - 1, n), 0.2, dtype=real, device="cuda"))
    f0 = ml.workspace[:n * (8 if prec == "f64" else 4)].view(real)
    assert bool((f0 == torch.tensor(1 / 3, dtype=real)).all()) == (not moments)
    ml.step(2)
    assert float((ml.populations()[0].reshape(19, n)[0] - 1 / 3).abs().max()) < 1e-6


@pytest.mark.parametrize("shape", [(20, 17, 13), (40, 16, 8)])
def test_more_planes_per_block_than_the_lattice_has(shape):
    lat, ref = _plain(shape, "f32"), _plain(shape, "f32")
    lat.set_step_form("auto", 2**31 - 1)
    lat.step(2)
    ref.step(2)
    assert all(torch.equal(a, b) for a, b in zip(lat.populations(), ref.populations()))
