"""The single-pass step of D2Q9 over populations (tau_g = 1, faces periodic or
mirrors, viscosities or densities that differ) on the GPU, at the sizes where it
can go wrong: lattices narrower than the halo, the edges of the 16 x 4 and 32 x 8
tiles, and the smallest lattice of the large tiles.

FP64 against the oracle to 1e-12 on every population and on C, mu, pt and rho;
16-bit storage with unit roundoff u (2^-11, 2^-8): against two passes of the
same arithmetic, where a stored f may fall to the other side of a rounding (2 u
of its deviation from rest, which is below an eighth of the largest population);
with mirrors, where two passes keep g in 16 bits and the single pass does not,
against FP64 to the roundings of the stored f and of the g read back (4 u).
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S
from dsm_helpers import compare, direction_map, gpu_fields, gpu_lattice, gpu_pops, oracle_params, \
    rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2504_19941_gb300 as P  # noqa: E402

Z = ("periodic", "periodic")
M = ("mirror", "mirror")
FACES = {"periodic": None, "mirror_y": Z + M + Z, "mirror_xy": M + M + Z}


def _case(shape, faces, contrast, seed=0):
    n = int(np.prod(shape))
    rng = np.random.default_rng(seed)
    sd = rng.uniform(-4.0, 1.0, n) if min(shape) < 8 else \
        S.sphere_sd(shape, [s / 3 for s in shape], min(shape) / 4).ravel()
    c1 = 0.5 + 0.5 * np.tanh(sd / 2.0)
    c2 = (0.5 + 0.3 * np.sin(np.arange(n) * 0.37) + S.perturbation(seed, n)) * (1 - c1)
    case = S.Case("tile2", "D2Q9", shape, sd, c2, theta_deg=70.0, g23=0.01, g12=0.01, alpha_s=1.0,
                  body=(1e-6, -2e-6, 0.0))
    case.tau2, case.tau3, case.faces = 1.0, 0.6, FACES[faces]
    if contrast:
        case.rho2, case.rho3 = 1.0, 0.5
    return case


@pytest.mark.parametrize("faces", list(FACES))
@pytest.mark.parametrize("shape,contrast", [((2, 2), False), ((3, 2), True), ((17, 5), False),
                                            ((33, 9), True), ((320, 257), False)])
def test_single_pass_matches_oracle(shape, contrast, faces):
    case = _case(shape, faces, contrast)
    steps = 3 if np.prod(shape) > 10000 else 8
    lat = gpu_lattice(case, "f64")
    lat.step(steps)
    p = oracle_params(case, O.D2Q9)
    c1 = O.solid_profile(case.solid_sd, case.alpha_s)
    f, g = O.lb_init(p, 2, c1, case.c2)
    f, g = O.lb_run(p, 2, c1, f, g, steps)
    errs = compare(gpu_fields(lat), O.lb_fields(p, 2, c1, f, g), ("C", "mu", "pt", "rho"))
    gf, gg = gpu_pops(lat, direction_map(O.D2Q9))
    errs["f"], errs["g"] = rel_err(gf, f), rel_err(gg, g)
    assert max(errs.values()) < 1e-12, errs


@pytest.mark.parametrize("prec,bits", [("f16", 11), ("bf16", 8)])
def test_single_pass_in_16_bit_storage(prec, bits):
    u = 2.0 ** -bits
    case = _case((45, 13), "periodic", True)
    one, two = gpu_lattice(case, prec), gpu_lattice(case, prec)
    two.set_step_form("two_pass")
    one.step(2)
    two.step(2)
    assert all(rel_err(a.cpu().numpy(), b.cpu().numpy()) < u / 4
               for a, b in zip(one.populations(), two.populations()))
    case = _case((45, 13), "mirror_y", True)
    one, ref = gpu_lattice(case, prec), gpu_lattice(case, "f64")
    one.step(2)
    ref.step(2)
    assert all(rel_err(a.cpu().numpy(), b.cpu().numpy()) < 4 * u
               for a, b in zip(one.populations(), ref.populations()))


@pytest.mark.parametrize("faces", list(FACES))
def test_other_forms_of_the_state(faces):
    # reads leave the trajectory alone; a checkpoint goes on bitwise, also into
    # a lattice that steps in two passes; populations in, and populations of g
    case = _case((33, 9), faces, False, 3)
    ref = gpu_lattice(case, "f64")
    ref.step(12)
    fr, gr = ref.populations()
    a = gpu_lattice(case, "f64")
    a.step(4)
    a.field("mu")
    a.populations()
    a.observables()
    a.step(2)
    st = a.state()
    a.step(6)
    assert torch.equal(a.populations()[0], fr) and torch.equal(a.populations()[1], gr)
    b = gpu_lattice(case, "f64")
    b.set_state(st)
    assert b.g_implicit == (faces == "periodic")
    b.step(6)
    assert torch.equal(b.populations()[0], fr) and torch.equal(b.populations()[1], gr)
    c = gpu_lattice(case, "f64")
    c.set_step_form("two_pass")
    c.set_state(st)
    c.step(2)
    c.set_step_form("auto")
    c.step(2)
    c.set_g_storage("populations")
    c.step(1)
    c.set_g_storage("auto")
    P._lib.dsm_step_moments(c.h)
    P._lib.dsm_step_collide(c.h)
    d = gpu_lattice(case, "f64")
    d.set_populations(*ref.populations())
    for x in (c, d, ref):
        x.step(3)
    fr, gr = (t.cpu().numpy() for t in ref.populations())
    fd, gd = (t.cpu().numpy() for t in d.populations())
    assert rel_err(fd, fr) < 1e-13 and rel_err(gd, gr) < 1e-13
    fc, gc = (t.cpu().numpy() for t in c.populations())
    assert rel_err(fc, fr) < 1e-13 and rel_err(gc, gr) < 1e-13
