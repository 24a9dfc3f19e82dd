"""FP64 lattices in 3D on moments, which takes 32768 nodes: the step, the reads (from
the next step's moments), other forms of the state, checkpoints and the split step
at ragged sizes and given runs of planes.  Every lattice says that its state is
held as moments, so that another rule for the sizes cannot empty these tests.

Against the oracle 1e-12 of each quantity's scale, velocities (cancelling sums)
5e-12 of the speed; the same operations in another order 1e-13.
"""
import numpy as np
import pytest

import oracle as O
from dsm_helpers import compare, direction_map, gpu_fields, gpu_lattice, gpu_pops, rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2504_19941_gb300 as P  # noqa: E402
from test_gpu_mom import _case, _oracle  # noqa: E402


def _on_moments(lat):
    return int(lat.state()[:32].view(torch.int32)[7]) == 2


@pytest.mark.parametrize("shape,zrun", [((33, 32, 32), 0), ((33, 33, 33), 5), ((66, 31, 17), 4),
                                        ((45, 41, 19), 19), ((31, 64, 41), 1), ((32, 8, 131), 0)])
def test_step_and_reads_match_oracle(shape, zrun):
    case = _case(shape)
    one, two = gpu_lattice(case, "f64"), gpu_lattice(case, "f64")
    one.set_step_form("auto", zrun)
    two.set_step_form("two_pass")
    steps = 3
    p, c1, f, g, kind = _oracle(case, steps)
    of = O.lb_fields(p, 2, c1, f, g)
    speed = max(np.abs(of[k]).max() for k in ("ux", "uy", "uz"))
    perm = direction_map(kind)
    for x in (one, two):
        x.step(steps)
        assert _on_moments(x)
        fl = gpu_fields(x)
        errs = compare(fl, of, ("C", "mu", "pt", "rho"))
        for k in ("ux", "uy", "uz"):
            errs[k] = np.abs(fl[k] - of[k]).max() / speed / 5.0
        ob = x.observables()
        u2 = of["ux"] ** 2 + of["uy"] ** 2 + of["uz"] ** 2
        errs["mass"] = abs(ob["mass_c2"] / of["C"].sum() - 1.0)
        errs["kinetic"] = abs(ob["kinetic"] / (0.5 * of["rho"] * u2).sum() - 1.0) / 10.0
        errs["max_u"] = abs(ob["max_u"] / np.sqrt(u2.max()) - 1.0) / 5.0
        gf, gg = gpu_pops(x, perm)
        errs["f"], errs["g"] = rel_err(gf, f), rel_err(gg, g)
        assert max(errs.values()) < 1e-12, errs
    # reads leave the trajectory alone, whatever they make
    fresh = gpu_lattice(case, "f64")
    fresh.set_step_form("auto", zrun)
    fresh.step(steps + 2)
    one.step(2)
    assert all(torch.equal(u, v) for u, v in zip(one.populations(), fresh.populations()))


@pytest.mark.parametrize("shape", [(33, 32, 32), (66, 31, 17)])
def test_other_forms_of_the_state(shape):
    case = _case(shape, 3)
    ref = gpu_lattice(case, "f64")
    ref.step(8)
    fr, gr = (t.cpu().numpy() for t in ref.populations())
    a = gpu_lattice(case, "f64")
    a.step(4)
    b = gpu_lattice(case, "f64")
    b.set_populations(*a.populations())
    b.step(2)
    assert _on_moments(b)
    b.set_g_storage("populations")
    b.step(1)
    assert not _on_moments(b)
    b.set_g_storage("auto")
    b.step(1)
    st = a.state()
    assert _on_moments(a)
    same, pops = gpu_lattice(case, "f64"), gpu_lattice(case, "f64", g_storage="populations")
    same.set_state(st)
    pops.set_state(st)
    split = gpu_lattice(case, "f64")
    for _ in range(8):
        P._lib.dsm_step_moments(split.h)
        P._lib.dsm_step_collide(split.h)
    assert _on_moments(split)
    for x in (a, same, pops):
        x.step(4)
    assert all(torch.equal(u, v) for u, v in zip(a.populations(), same.populations()))
    for x in (b, pops, split):
        fx, gx = (t.cpu().numpy() for t in x.populations())
        assert rel_err(fx, fr) < 1e-13 and rel_err(gx, gr) < 1e-13
