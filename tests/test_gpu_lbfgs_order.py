"""The minimiser's iterates, to the bit.  L-BFGS amplifies the last place of an
energy or of a dot product into the iterates (a change of one unit in E moves
the point after 25 iterations by up to 1e-2), so every sum of the minimiser is
taken in one fixed order, and these iterates are part of its result.

golden/lbfgs_iterates.txt holds, per case, the SHA-256 of x, E as a hexadecimal
double, iterations and evaluations, as the library has given them since its
first release on a GB300.  The inputs use only correctly rounded operations, so
they are the same bits on every host.  The cases: vectors that are and are not a
multiple of four long, shorter and longer than one and four strides of the
vector kernels (155648 elements), more stored pairs than one pass of the update
takes (m > 10), each constraint, the solid as the active field, and N fluids.
"""
import hashlib
import math
import os

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_2504_19941_gb300 as P  # noqa: E402
from paper_2504_19941_gb300.energy import (FreeEnergy, FreeEnergyMulti, lbfgs,  # noqa: E402
                                           lbfgs_multi)

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "lbfgs_iterates.txt")
Z = ("periodic", "periodic")

# shape, iterations, arguments
CASES = {
    "3d_kcs": ((33, 18, 21), 25, dict(kcs=1e-2)),
    "3d_dP": ((48, 40, 36), 20, dict(dP=2e-3)),
    "3d_long": ((96, 96, 81), 25, dict(kcs=1e-2)),
    "3d_branch": ((96, 96, 81), 25, dict(kcs=1e-2, seed=1)),  # a last place decides a step
    "3d_mirror": ((31, 24, 19), 20, dict(kcs=2e-2, faces=("mirror", "mirror") + Z + Z)),
    "2d_kcs": ((97, 70), 40, dict(kcs=1e-2)),
    "2d_m14": ((64, 50), 40, dict(kcs=1e-2, m=14)),
    "2d_m3": ((320, 401), 20, dict(kcs=1e-2, m=3)),
    "solid": ((24, 20, 17), 20, dict(active=1)),
    "gravity": ((40, 33), 20, dict(dP=1e-3, fg=1e-4)),
    "multi": ((32, 24, 21), 20, dict(nfluid=3)),
}


def _smooth(s):  # from 0 to 1 over a few nodes
    return 0.5 + 0.5 * s / np.sqrt(1.0 + s * s)


def _fields(shape, seed):
    rng = np.random.default_rng(seed)
    X = np.meshgrid(*[np.arange(n, dtype=np.float64) for n in reversed(shape)], indexing="ij")
    h = X[0]
    c1 = _smooth(4.0 - h)
    r = np.sqrt(sum((x - (7.0 if a == 0 else n / 2.0)) ** 2
                    for a, (x, n) in enumerate(zip(X, reversed(shape)))))
    c2 = _smooth(0.25 * min(shape) - r) * (1.0 - c1)
    c2 = c2 + 1e-3 * (rng.random(c2.shape) - 0.5)
    return c1.astype(np.float32).ravel(), c2.astype(np.float32).ravel()


def _run(name):
    shape, iters, kw = CASES[name]
    kw = dict(kw)
    dev = "cuda"
    c1, c2 = _fields(shape, kw.pop("seed", len(name)))
    p = P.make_params("D2Q9" if len(shape) == 2 else "D3Q19", shape, "f32", theta_deg=110.0,
                      g23=0.9375, g12=1.0, faces=kw.pop("faces", None), beta=0.5)
    t1, t2 = torch.as_tensor(c1, device=dev), torch.as_tensor(c2, device=dev)
    if kw.pop("nfluid", 0):
        left = np.arange(c2.size) % shape[0] < shape[0] // 2
        C = torch.as_tensor(np.stack([c2 * left, c2 * ~left]), device=dev)
        V0 = [math.fsum(c2[left]), math.fsum(c2[~left])]
        x, E, info = lbfgs_multi(FreeEnergyMulti(p, 3, [0.02, 0.03, 0.025, 0.035]), C, t1,
                                 kcs=[1e-2, 1e-2], V0=V0, tol=0.0, max_iter=iters)
    elif kw.get("active") == 1:
        mask = torch.as_tensor((c1 > 0.5).astype(np.uint8), device=dev)
        x, E, info = lbfgs(FreeEnergy(p), t1, t2, mask=mask, tol=0.0, max_iter=iters, **kw)
    else:
        V0 = 0.999 * math.fsum(c2) if "kcs" in kw else 0.0
        x, E, info = lbfgs(FreeEnergy(p), t2, t1, V0=V0, tol=0.0, max_iter=iters, **kw)
    bits = hashlib.sha256(x.cpu().numpy().tobytes()).hexdigest()
    return f"{name} {bits} {float(E).hex()} {info['iterations']} {info['evaluations']}"


@pytest.mark.parametrize("name", list(CASES))
def test_iterates_are_the_recorded_ones(name):
    with open(GOLDEN) as f:
        want = {line.split()[0]: line.strip() for line in f}
    assert _run(name) == want[name]
