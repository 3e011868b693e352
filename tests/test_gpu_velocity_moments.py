"""Velocity moments per shell against numpy's float64: few and many shells
(32 lane copies of the sums down to one), ragged counts, particles on the
axis and at the centre, shells that hold nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


@pytest.mark.parametrize("prec", ["fp32c", "fp64"])
@pytest.mark.parametrize("n,nshell", [(1, 1), (257, 8), (40_003, 1), (40_003, 37), (40_003, 200), (40_003, 1024)])
def test_moments_match_float64(prec, n, nshell):
    from paper_1207_6403_gb300 import m2m
    P = I.make_problem("plain-fp64", n=n, precision=prec, with_target=False)
    dt = np.float32 if prec == "fp32c" else np.float64
    rng = np.random.default_rng(n + nshell)
    P.w0[:] = rng.random(n) / n
    if n > 100:
        P.pos[:2, 10:20] = 0.0           # on the axis
        P.pos[:, 20:22] = 0.0            # at the centre
    e = np.concatenate([[0.0], np.geomspace(1e-4, 50.0, nshell) ** 2])
    ctx = m2m.from_problem(P, prec, targets=False)
    got = ctx.m2m_velocity_moments(e)
    again = ctx.m2m_velocity_moments(e[: max(2, len(e) // 2)])      # fewer shells in the kept buffer
    ctx.m2m_free()
    x, v = P.pos.astype(dt), P.vel.astype(dt)
    k = np.searchsorted(e, ((x[0] * x[0] + x[1] * x[1]) + x[2] * x[2]).astype(np.float64), side="right") - 1
    ok = (k >= 0) & (k < nshell)
    x, v = x.astype(np.float64), v.astype(np.float64)
    r2, R2 = (x * x).sum(0), x[0] ** 2 + x[1] ** 2
    with np.errstate(invalid="ignore", divide="ignore"):
        vr2 = np.where(r2 > 0, (x * v).sum(0) ** 2 / r2, 0.0)
        vp2 = np.where(R2 > 0, (x[0] * v[1] - x[1] * v[0]) ** 2 / R2, 0.0)
    v2 = (v * v).sum(0)
    want, scale = np.zeros((nshell, 4)), np.zeros(nshell)
    for c, t in enumerate((np.ones(n), vr2, v2 - vr2 - vp2, vp2)):
        np.add.at(want[:, c], k[ok], (P.w0 * t)[ok])
    np.add.at(scale, k[ok], (P.w0 * (1.0 + v2))[ok])
    # n roundings of a double sum and a few of each term
    tol = (n + 16) * 2.0 ** -53 * scale[:, None]
    assert np.all(np.abs(got - want) <= tol)
    m = again.shape[0]
    assert np.all(np.abs(again - want[:m]) <= tol[:m])
