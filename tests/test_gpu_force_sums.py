"""The exact force sums of bodies with many nodes: the volume-integral force of one step
from a prescribed state against the same sum in extended precision.  One term per solid
node, all of one sign, is what fills the fixed-point words fastest."""
import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu

WT = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]


@pytest.mark.parametrize("u", [(0.04, 0.03), (-0.04, -0.03)])
@pytest.mark.parametrize("uniform", [False, True])
@pytest.mark.parametrize("length", [60.0, 200.0])
def test_volume_integral_of_a_large_body(length, uniform, u):
    """2,800 and 31,400 solid nodes in a stream against a body at rest: equal terms at
    every node, or terms of random low bits."""
    nx, ny = 2 * int(length) + 13, int(length) + 31
    w = W.Workload(name="large", nx=nx, ny=ny, dtype="f64", collision="trt", tau_plus=0.6, u_in=u,
                   bc=("periodic",) * 4, steps=1,
                   body=W.Body("disk", length=length, x_c=0.5 * nx + 0.2, y_c=0.5 * ny - 0.3))
    lat = V.Lattice(V.config_of(w))
    lat.set_body(V.body_of(w))
    cu = CX * u[0] + CY * u[1]
    f = np.broadcast_to(WT * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u[0] ** 2 + u[1] ** 2)), (9, ny, nx)).copy()
    if not uniform:
        f *= 1 + 0.02 * np.random.default_rng(4).uniform(-1, 1, f.shape)
    lat.set_state(f, f, post_collision=False)
    f = lat.get_f()
    lat.step(1)
    got = lat.force_angot()
    solid = lat.get_mask() != 0
    fl = f[:, solid].astype(np.longdouble)
    k = np.longdouble(0.5) / np.longdouble(w.eta)
    jx, jy = ((c[:, :, 0] * fl).sum(0) * 2 * k / (1 + k) for c in (CX, CY))
    y, x = np.nonzero(solid)
    rx, ry = x - np.longdouble(w.body.x_c), y - np.longdouble(w.body.y_c)
    # per node: the populations read back, eight sums of them and three products are
    # rounded, each within half a unit of the sum of the populations' sizes (the
    # torque's two products and their difference on top)
    eps = np.longdouble(2.0) ** -53
    size = 2 * np.abs(fl).sum(0)
    assert solid.sum() > 0.7 * length ** 2
    for g, terms, arm in ((got[0], jx, 1), (got[1], jy, 1), (got[2], rx * jy - ry * jx, np.abs(rx) + np.abs(ry))):
        assert abs(g - terms.sum()) <= 16 * eps * (size * arm).sum()
