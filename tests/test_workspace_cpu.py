"""Workspace bytes callers have been asked for stay what they were: a lattice that
fitted the device before it stepped on moments still does.  The figures are those
of the library before that step."""
import pytest

import paper_2504_19941_gb300 as P
from paper_2504_19941_gb300 import _lib


@pytest.mark.parametrize("prec,shape,nfluid,nbytes", [
    ("f32", (32, 8, 64), 2, 4301056), ("f32", (32, 32, 32), 3, 9056512),
    ("f64", (64, 64, 64), 4, 154583296), ("f64", (101, 101, 101), 3, 538180864),
    ("f32", (45, 13, 7), 3, 1187840), ("f32", (24, 16, 8), 3, 590080), ("f64", (33, 8, 1), 4, 211456)])
def test_lattices_of_several_fluids(prec, shape, nfluid, nbytes):
    p = P.make_params("D3Q19", shape, prec, theta_deg=90.0)
    assert _lib.dsm_ml_workspace_bytes(p, nfluid) <= nbytes


@pytest.mark.parametrize("shape,m,nbytes", [((16, 16, 16), 10, 423424), ((64, 64, 64), 10, 25408512),
                                            ((128, 128, 128), 10, 201569280),
                                            ((64, 64, 64), 20, 46574848)])
def test_the_minimiser(shape, m, nbytes):
    p = P.make_params("D3Q19", shape, "f32", theta_deg=90.0)
    assert _lib.dsm_lbfgs_workspace_bytes(p, m) <= nbytes
