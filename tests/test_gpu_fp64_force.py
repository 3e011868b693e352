"""The FP64 force's quotient where rounding it is hardest: GM / ((r s) s) an
extreme distance from the middle of two doubles, against IEEE division."""
import numpy as np
import pytest

from oracle import m2m as O
from paper_1207_6403_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# numerator and divisor (integers below 2^53, scaled) whose quotient is within
# 2^-53 ulp or so of a midpoint: odd M with M b = -+1 mod 2^53 (2^54)
PAIRS = [("0x1.4671f637437cp+0", "0x1.ff6bb2ac620e9p+0"), ("0x1.8dbd55537f9a4p+0", "0x1.ffccd2cd33919p+0"),
         ("0x1.b43f361db3f45p+0", "0x1.ff13300059aa7p+0"), ("0x1.39a48e5b64367p+0", "0x1.ffc4f2b9db4efp+0"),
         ("0x1.070d5523fe242p+0", "0x1.ff8c80f0258bbp+0"), ("0x1.fd7567188b527p+0", "0x1.fff68f4e8d1e7p+0")]
DT = 2.0 ** -20


def _position(GM, b, rng):
    """r and a with (r (r + a)) (r + a) = b in double, at which one ulp of the
    quotient reaches the velocity after a step."""
    for _ in range(100_000):
        a = float(rng.uniform(0.1, 1.0))
        r = 0.5
        for _ in range(60):
            r -= (r * (r + a) ** 2 - b) / ((r + a) * (3 * r + a))
        for k in range(-6, 7):
            q = r + k * np.spacing(r)
            s = q + a
            if (q * s) * s != b:
                continue
            h, f = DT / 2, GM / b
            v = []
            for f1 in (f, np.nextafter(f, 0.0), np.nextafter(f, 9.0)):
                v1 = h * -(f1 * q)
                x = q + DT * v1
                s2 = x + a
                v.append(v1 + h * -(GM / ((x * s2) * s2) * x))
            if v[1] != v[0] and v[2] != v[0]:
                return q, a
    raise AssertionError("no position found")


@pytest.mark.parametrize("pair", PAIRS)
def test_force_quotient_is_ieee_division(pair):
    from paper_1207_6403_gb300 import m2m as B
    GM, b = (float.fromhex(v) for v in pair)
    r, a = _position(GM, b, np.random.default_rng(1))
    comps = [I.PotentialComponent("hernquist", (GM, a))]
    P = I.make_problem("plain-fp64", n=3, precision="fp64", with_target=False)
    P.pos = np.array([[r, 0.0, 0.0], [0.0, r, 0.0], [0.0, 0.0, -r]]).T.copy()
    P.vel = np.zeros((3, 3))
    P.potential, P.dt = comps, DT
    P.Y = P.sigma = None
    ctx = B.from_problem(P, "fp64", targets=False)
    ctx.m2m_push(1)
    g = ctx.state()
    ctx.m2m_free()
    for k, q in zip(("x", "y", "z", "vx", "vy", "vz"), O.kdk(*P.pos, *P.vel, comps, DT)):
        np.testing.assert_array_equal(g[k], q, err_msg=k)
