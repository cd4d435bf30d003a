"""Momentum of FP64 lattices over many collisions: in an empty periodic lattice the mean
momentum of a node stays, however slowly the odd moments relax."""
import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]


# odd rates s- of 0.03, 0.17, 0.26 and 0.46 (below the line at which the form of the
# collision changes), 0.53, 0.95 and 1.54
@pytest.mark.parametrize("collision,tau", [("trt", 0.505), ("trt", 0.53), ("trt", 0.55), ("trt", 0.6),
                                           ("trt", 0.62), ("trt", 0.8), ("bgk", 0.65)])
def test_fp64_momentum_has_no_drift(collision, tau):
    n, u, steps = 256, (0.04, -0.03), 50
    w = W.Workload(name="box", nx=n, ny=n, dtype="f64", collision=collision, tau_plus=tau, u_in=(0.0, 0.0),
                   bc=("periodic",) * 4, body=W.Body("none"), steps=1)
    lat = V.Lattice(V.config_of(w))
    lat.set_body(V.body_of(w))
    cu = CX * u[0] + CY * u[1]
    f = WT * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u[0] ** 2 + u[1] ** 2))
    f = f * (1 + 1e-3 * np.random.default_rng(2).uniform(-1, 1, (9, n, n)))
    lat.set_state(f, f, post_collision=False)

    def momentum():
        g = lat.get_f().astype(np.longdouble)
        return [(c * g).sum() / n ** 2 for c in (CX, CY)]

    before = momentum()
    lat.step(steps)
    # a coefficient of the odd part rounded once may move the momentum by u 2^-54 in
    # every step; exact coefficients leave roundings that average out, to less than a
    # tenth of that per step over the nodes, beside the read-back's own (some 1e-17
    # per node, 65536 nodes)
    for a, b, v in zip(before, momentum(), u):
        assert abs(a - b) <= 0.1 * steps * abs(v) * 2.0 ** -54 + 1e-18
