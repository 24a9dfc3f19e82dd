"""The step on moments (every relaxation time 1, equal densities, periodic
faces) on the GPU, at the sizes where it can go wrong: single nodes, lattices
narrower than the stencil's halo, edges of the 32 x 8 tiles and of the runs of
planes, and the smallest lattice of the large 2D tiles.

FP64 against the oracle to 1e-12 on every population and on C, mu, pt and rho.
The two-pass form and
the single pass are the same operations in another order: FP64 equal to 1e-13.
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


def _case(shape, seed=0):
    n = int(np.prod(shape))
    d = len(shape)
    rng = np.random.default_rng(seed)
    sd = rng.uniform(-4.0, 1.0, n) if min(shape) < 8 else \
        S.sphere_sd(shape, [s / 3 for s in shape], min(shape) / 4).ravel()
    c1 = 0.5 + 0.5 * np.tanh(sd / 2.0)
    c2 = (0.5 + 0.3 * np.sin(np.arange(n) * 0.37) + S.perturbation(seed, n)) * (1 - c1)
    return S.Case("mom", "D2Q9" if d == 2 else "D3Q19", shape, sd, c2, theta_deg=70.0, g23=0.01,
                  g12=0.01, alpha_s=1.0, body=(1e-6, -2e-6, 0.0 if d == 2 else 3e-6))


def _oracle(case, steps):
    kind = O.D2Q9 if case.lattice == "D2Q9" else O.D3Q19
    p = oracle_params(case, kind)
    c1 = O.solid_profile(case.solid_sd, case.alpha_s)
    f, g = O.lb_init(p, 2, c1, case.c2)
    return p, c1, *O.lb_run(p, 2, c1, f, g, steps), kind


SHAPES = [((1, 1, 1), 0), ((2, 3, 1), 0), ((31, 8, 3), 1), ((33, 9, 5), 2), ((66, 17, 9), 4),
          ((1, 1), 0), ((3, 2), 0), ((33, 9), 0), ((320, 257), 0)]


@pytest.mark.parametrize("shape,zrun", SHAPES)
def test_step_on_moments_matches_oracle(shape, zrun):
    case = _case(shape)
    steps = 3 if np.prod(shape) > 10000 else 8
    lat, two = gpu_lattice(case, "f64"), gpu_lattice(case, "f64")
    lat.set_step_form("auto", zrun)
    two.set_step_form("two_pass")
    lat.step(steps)
    two.step(steps)
    p, c1, f, g, kind = _oracle(case, steps)
    perm = direction_map(kind)
    of = O.lb_fields(p, 2, c1, f, g)
    for x in (lat, two):
        gfl = gpu_fields(x)
        errs = compare(gfl, of, ("C", "mu", "pt", "rho"))
        gf, gg = gpu_pops(x, perm)
        errs["f"], errs["g"] = rel_err(gf, f), rel_err(gg, g)
        assert max(errs.values()) < 1e-12, errs
    a, b = lat.populations(), two.populations()
    assert all(rel_err(u.cpu().numpy(), v.cpu().numpy()) < 1e-13 for u, v in zip(a, b))


@pytest.mark.parametrize("shape", [(33, 9, 5), (33, 9)])
def test_moments_and_other_forms_of_the_state(shape):
    # populations in, populations form mid-run, and a checkpoint restored into a
    # lattice of the same kind and into one that keeps its state otherwise
    case = _case(shape, 3)
    ref = gpu_lattice(case, "f64")
    ref.step(12)
    fr, gr = (t.cpu().numpy() for t in ref.populations())
    a = gpu_lattice(case, "f64")
    a.step(4)
    b = gpu_lattice(case, "f64")
    b.set_populations(*a.populations())
    assert not b.g_implicit
    b.step(4)
    assert b.g_implicit
    b.set_g_storage("populations")
    b.step(2)
    b.set_g_storage("auto")
    b.step(2)
    fb, gb = (t.cpu().numpy() for t in b.populations())
    assert rel_err(fb, fr) < 1e-13 and rel_err(gb, gr) < 1e-13
    st = a.state()
    same = gpu_lattice(case, "f64")
    same.set_state(st)
    pops = gpu_lattice(case, "f64", g_storage="populations")
    pops.set_state(st)
    assert same.g_implicit and not pops.g_implicit
    a.step(8)
    same.step(8)
    pops.step(8)
    assert all(torch.equal(u, v) for u, v in zip(a.populations(), same.populations()))
    fp, gp = (t.cpu().numpy() for t in pops.populations())
    assert rel_err(fp, fr) < 1e-13 and rel_err(gp, gr) < 1e-13
    # the split step on moments is the two-pass step
    s = gpu_lattice(case, "f64")
    for _ in range(12):
        P._lib.dsm_step_moments(s.h)
        P._lib.dsm_step_collide(s.h)
    fs, gs = (t.cpu().numpy() for t in s.populations())
    assert rel_err(fs, fr) < 1e-13 and rel_err(gs, gr) < 1e-13
