"""Velocity moments of particles whose squares leave the double range although
their velocities do not: close to the axis, far out, slow and fast."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


# one particle a call: position and velocity scales, and the same particle
# turned onto the axes; v_r and v_phi squared stay normal numbers
@pytest.mark.parametrize("rs,vs", [(1e-145, 1.0), (1e-120, 1e-30), (1e-60, 1e-110), (1e-45, 1e-120), (1e-45, 1e140),
                                   (1e-30, 1e-150), (1.0, 1e-150), (1.0, 0.0), (1.0, 1e150), (1e45, 1e150),
                                   (1e60, 1e100), (1e100, 1e-140), (1e145, 1.0), (1e145, 1e150)])
@pytest.mark.parametrize("turn", [0, 1, 2])
def test_one_particle_at_every_scale(rs, vs, turn):
    from paper_1207_6403_gb300 import m2m
    P = I.make_problem("plain-fp64", n=1, precision="fp64", with_target=False)
    x, v = np.array([0.3, -0.4, 1.2]) * rs, np.array([0.7, 0.9, -0.2]) * vs
    if turn == 1:
        x[2] = 0.0                                # in the plane
    if turn == 2:
        x[0] *= 1e-3                              # near an axis of the plane
    P.pos, P.vel, P.w0[:] = x[:, None].copy(), v[:, None].copy(), 0.625
    ctx = m2m.from_problem(P, "fp64", targets=False)
    got = ctx.m2m_velocity_moments(np.array([0.0, 1e300]))[0]
    ctx.m2m_free()
    x, v = x.astype(np.longdouble), v.astype(np.longdouble)
    vr2 = (x * v).sum() ** 2 / (x * x).sum()
    vp2 = (x[0] * v[1] - x[1] * v[0]) ** 2 / (x[0] ** 2 + x[1] ** 2)
    v2 = (v * v).sum()
    want = 0.625 * np.array([1.0, vr2, v2 - vr2 - vp2, vp2])
    # the few roundings of each term, x.v and x vy - y vx cancelling to a tenth at worst
    tol = 64 * 2.0 ** -53
    assert got[0] == want[0]
    assert abs(got[1] - want[1]) <= tol * want[1] and abs(got[3] - want[3]) <= tol * want[3]
    assert abs(got[2] - want[2]) <= tol * 0.625 * v2
