"""A moving disk, whose every block updates the body from the previous step's sums:
runs replayed from step graphs, single-step calls and steps queued one by one (SIM on
some steps only) end bit-identical, and a disk that would leave the lattice stays where
it was in all of them, flagged."""
import numpy as np
import pytest

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def falling(dtype, est, y=60.0, g=4e-4):
    body = W.Body("disk", length=13.0, x_c=31.3, y_c=y, moving=True, density_ratio=1.2,
                  gravity=(2e-5, -g), estimator=est)
    return W.Workload(name="fall", nx=150, ny=90, dtype=dtype, collision="trt", tau_plus=0.6, u_in=(0.0, 0.0),
                      bc=("noslip",) * 4, body=body, steps=1)


def lattice(w, **over):
    lat = V.Lattice(V.config_of(w, **over))
    lat.set_body(V.body_of(w))
    return lat


def same(a, b, n):
    np.testing.assert_array_equal(a.get_f(), b.get_f())
    np.testing.assert_array_equal(a.get_body(), b.get_body())
    np.testing.assert_array_equal(a.get_mask(), b.get_mask())
    for est in (V.MEM, V.SIM, V.ANGOT):
        np.testing.assert_array_equal(a.history(est, n), b.history(est, n))
    for p, q in zip(a.sums(), b.sums()):
        np.testing.assert_array_equal(p, q)


@pytest.mark.parametrize("dtype", ["f64", "f32", "f16sr"])
@pytest.mark.parametrize("est", ["mem", "sim"])
def test_runs_equal_single_steps(dtype, est):
    w = falling(dtype, est)
    runs, single = lattice(w), lattice(w)
    for n in (1, 2, 3, 32, 7):
        runs.step(n)
    for _ in range(45):
        single.step(1)
    same(runs, single, 45)
    runs.check()
    assert runs.get_body()[1] < 60.0


def test_steps_queued_one_by_one():
    """SIM on every second step: no graphs, three sets of sums in turn over one call.
    The flow and the MEM-driven body are those of a lattice with SIM on every step."""
    w = falling("f32", "mem")
    sparse, every = lattice(w, sim_every=2), lattice(w)
    sparse.step(14)
    sparse.step(11)
    every.step(25)
    np.testing.assert_array_equal(sparse.get_f(), every.get_f())
    np.testing.assert_array_equal(sparse.get_body(), every.get_body())
    np.testing.assert_array_equal(sparse.history(V.MEM, 25), every.history(V.MEM, 25))
    s, e = sparse.history(V.SIM, 25), every.history(V.SIM, 25)
    np.testing.assert_array_equal(s[::2], e[::2])
    assert np.isnan(s[1::2]).all()


def test_a_disk_that_would_leave_the_lattice_stays_and_is_flagged():
    """A heavy disk thrown at the lower wall, 1.5 nodes from leaving the lattice at 0.9
    nodes per step: it leaves in the second step."""
    w = falling("f32", "mem", y=8.0)
    body = V.body_of(w)
    body.u[1] = -0.9
    body.density_ratio = 50.0
    runs, single = V.Lattice(V.config_of(w)), V.Lattice(V.config_of(w))
    for lat in (runs, single):
        lat.set_body(body)
    runs.step(7)
    for _ in range(7):
        single.step(1)
    same(runs, single, 7)
    y = runs.get_body()[1]
    assert 6.5 <= y < 8.0
    with pytest.raises(V.VplbmError) as err:
        runs.check()
    assert err.value.status == V.EUNSTABLE
