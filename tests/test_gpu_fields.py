"""The macroscopic fields of the read-back against extended-precision sums of the
populations it belongs to: every storage form, small offsets (summed as integers on
the device), large ones and a body (the general form), wide and ragged lattices."""
import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])[:, None, None]
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])[:, None, None]


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16", "bf16", "f16sr"])
@pytest.mark.parametrize("shape", [(131, 40), (257, 7), (300, 3)])
@pytest.mark.parametrize("lo,hi", [(0.10, 0.12), (0.05, 0.4), (0.4, 1.3)])
@pytest.mark.parametrize("post", [False, True])
def test_fields_are_the_moments_of_the_populations(dtype, shape, lo, hi, post):
    nx, ny = shape
    body = W.Body("disk", length=9.0, x_c=30.2, y_c=0.5 * ny) if ny > 20 else W.Body("none")
    w = W.Workload(name="fields", nx=nx, ny=ny, dtype=dtype, collision="trt", tau_plus=0.7, u_in=(0.05, 0.01),
                   bc=("inlet", "outlet", "symmetry", "noslip"), body=body, steps=1,
                   body_force=(3e-5, -1e-5), u_ref=(0.05, 0.0))
    lat = V.Lattice(V.config_of(w))
    lat.set_body(V.body_of(w))
    f = W.random_field(3, (9, ny, nx), lo=lo, hi=hi)
    lat.set_state(f, f, post_collision=post)
    f = lat.get_f().astype(np.longdouble)
    rho, ux, uy = lat.get_fields()
    r = f.sum(0)
    jx = (CX * f).sum(0) + np.longdouble(0.5 * 3e-5)
    jy = (CY * f).sum(0) + np.longdouble(0.5 * -1e-5)
    k = lat.get_mask() * np.longdouble(0.5 / w.eta)
    # the populations read back are rounded once (2^-53 each), the fields to
    # FP64 with a reciprocal and a product (two units)
    eps = np.longdouble(2.0) ** -53
    size = np.abs(f).sum(0)
    assert np.all(np.abs(rho - r) <= eps * (size + 2 * r))
    for got, j in ((ux, jx), (uy, jy)):
        ref = j / (r * (1 + k))
        assert np.all(np.abs(got - ref) <= eps * (2 * size / (r * (1 + k)) * (1 + np.abs(ref)) + 8 * np.abs(ref)))


@pytest.mark.parametrize("dtype", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("force", [(7.5, -7.5), (8.5, 0.1), (0.1, -11.5), (25.0, -40.0), (1e30, 1e-30)])
def test_fields_under_a_large_body_force(dtype, force):
    """Half the body force is part of the momentum, whatever its size."""
    nx, ny = 131, 9
    w = W.Workload(name="force", nx=nx, ny=ny, dtype=dtype, collision="trt", tau_plus=0.7, u_in=(0.05, 0.01),
                   bc=("inlet", "outlet", "symmetry", "noslip"), body=W.Body("none"), steps=1,
                   body_force=force, u_ref=(0.05, 0.0))
    lat = V.Lattice(V.config_of(w))
    lat.set_body(V.body_of(w))
    f = W.random_field(3, (9, ny, nx), lo=0.10, hi=0.12)
    lat.set_state(f, f, post_collision=False)
    f = lat.get_f().astype(np.longdouble)
    rho, ux, uy = lat.get_fields()
    r = f.sum(0)
    eps = np.longdouble(2.0) ** -53
    size = np.abs(f).sum(0)
    assert np.all(np.abs(rho - r) <= eps * (size + 2 * r))
    for got, c, g in ((ux, CX, force[0]), (uy, CY, force[1])):
        ref = ((c * f).sum(0) + np.longdouble(0.5) * np.longdouble(g)) / r
        # as above, and half the force added and rounded once more
        assert np.all(np.abs(got - ref) <= eps * (2 * size / r * (1 + np.abs(ref)) + 8 * np.abs(ref)))
