"""A state's form when it changes hands: checkpoints restored into lattices of
other relaxation times or faces, which hold and step their state otherwise.
Everything compared here is the same operations on the same numbers: equal bits.
"""
import pytest

import synthetic as S
from dsm_helpers import gpu_lattice

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_19941_gb300 import _lib  # noqa: E402


def _case(shape=(45, 13), **kw):
    sd = S.sphere_sd(shape, [s / 3 for s in shape], 4.0)
    c2 = S.drop_c2(shape, [s / 2 for s in shape], 4.0, 1.0, sd, 1.0).ravel()
    case = S.Case("forms", "D2Q9" if len(shape) == 2 else "D3Q19", shape, sd.ravel(),
                  c2 + S.perturbation(3, sd.size), theta_deg=70.0, g23=0.01, g12=0.01,
                  alpha_s=1.0, body=(1e-6, -2e-6, 0.0))
    for k, v in kw.items():
        setattr(case, k, v)
    return case


def _equal(a, b):
    return all(torch.equal(u, v) for u, v in zip(a.populations(), b.populations()))


def _batch(lat, n):
    nb = _lib.dsm_batch_scratch_bytes([lat.h])
    _lib.dsm_batch_step([lat.h], [n], torch.empty(nb, dtype=torch.uint8, device="cuda"), nb)


def _quads():
    # held as f and quads (A, C, u) by a lattice with two viscosities
    donor = gpu_lattice(_case(tau3=0.6), "f64")
    donor.step(4)
    return donor.state()


def _restored(st, **kw):
    lat = gpu_lattice(_case(**kw), "f64")
    lat.set_state(st)
    return lat


def test_a_batched_step_on_moments_ends_the_quads():
    st = _quads()
    ref, lat = _restored(st), _restored(st)
    ref.step(1)
    _batch(lat, 1)
    assert _equal(lat, ref)
    assert _equal(_restored(lat.state()), ref)


def test_a_new_fluid_on_moments_ends_the_quads():
    lat, new = gpu_lattice(_case(), "f64"), gpu_lattice(_case(), "f64")
    lat.set_step_form("two_pass")
    new.set_step_form("two_pass")
    lat.set_state(_quads())
    for x in (lat, new):
        x.set_fluid(torch.as_tensor(_case().c2, dtype=x.real, device="cuda"))
        x.field("mu")
        x.step(1)
    assert _equal(lat, new)


@pytest.mark.parametrize("kw", [dict(tau_g=0.8),
                                dict(faces=("periodic",) * 2 + ("wall",) * 2 + ("periodic",) * 2)])
@pytest.mark.parametrize("prec", ["f64", "f16"])
def test_quads_into_a_lattice_without_that_step(prec, kw):
    # tau_g != 1 and walls keep g as populations and step in two passes
    donor = gpu_lattice(_case(tau3=0.6), prec)
    donor.step(4)
    lat, ref = gpu_lattice(_case(**kw), prec), gpu_lattice(_case(**kw), prec)
    lat.set_state(donor.state())
    ref.set_populations(*donor.populations())
    assert not lat.g_implicit and lat.observables()["step"] == 4
    for _ in range(2):
        # (g_eq formed at its nodes and read back: in 16 bits equal to a rounding)
        for a, b in zip(lat.populations(), ref.populations()):
            assert float((a - b).abs().max()) <= (1e-14 if prec == "f64" else 2.0 ** -11)
        lat.step(3)
        ref.step(3)


@pytest.mark.parametrize("shape", [(45, 13), (33, 9, 5)])
def test_a_state_at_rest_keeps_its_storage_form(shape):
    # dsm_get_g_storage: g of a new fluid are populations until the first step
    lat, other = gpu_lattice(_case(shape), "f32"), gpu_lattice(_case(shape), "f32")
    other.step(2)
    other.set_state(lat.state())
    assert not lat.g_implicit and not other.g_implicit
    lat.step(2)
    other.step(2)
    assert other.g_implicit and _equal(lat, other)


@pytest.mark.parametrize("shape,prec", [((33, 9, 5), "f32"), ((45, 13), "f32"), ((45, 13), "f64"),
                                        ((40, 16, 8), "f16")])
def test_a_read_does_not_latch_what_the_next_step_would_meet(shape, prec):
    # a body force whose step overflows, read and taken back: the state is sound
    lat, twin = gpu_lattice(_case(shape), prec), gpu_lattice(_case(shape), prec)
    lat.step(3)
    twin.step(3)
    lat.set_body_force((1e200 if prec == "f64" else 1e30, 0.0, 0.0))
    lat.field("pt")
    assert float(lat.field("ux").abs().max()) > 1e20  # (its square overflows)
    for x in (lat, twin):
        x.set_body_force((1e-6, 0.0, 0.0))
    assert lat.observables()["nonfinite"] == 0
    lat.step(2)
    twin.step(2)
    assert lat.observables() == twin.observables() and _equal(lat, twin)
