"""ln(w/w_hat) over a long FP64 call: it follows the stored weights, however
many steps the call has."""
import numpy as np
import pytest

from paper_1207_6403_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# Without data the weights obey L_(t+1) = L_t - k (L_t + c), L = ln(w/w_hat),
# k = eps dt mu, which leaves L = -c to (1 - k)^4000 (4e-18 of the start at
# worst here).  A weight stops moving where |d| = k |L + c| is less than half
# an ulp of it, so L ends within 2^-53/k of -c, plus what the step's logarithm
# is off (two roundings, of the ratio and of the result); the rounding of a
# weight on the way decays with k.
@pytest.mark.parametrize("name", ["plain-fp64", "moving-priors", "flat-log", "ifu-lut"])
@pytest.mark.parametrize("k", [0.1, 0.01])
@pytest.mark.parametrize("n", [37, 2000])
def test_long_call_ends_where_the_entropy_does(name, k, n):
    from paper_1207_6403_gb300 import m2m as B
    P = I.make_problem(name, n=n, precision="fp64", with_target=False)
    rng = np.random.default_rng(n)
    P.what0 = np.exp(0.2 * rng.normal(size=n)) / n
    P.w0 = P.what0 * np.exp(0.3 * rng.normal(size=n))
    P.Y, P.sigma = np.ones(P.nobs), np.zeros(P.nobs)       # no observable counts
    P.prior = I.PriorSpec("flat")
    P.mu, P.eps = 10.0, k / (10.0 * P.dt)
    ctx = B.from_problem(P, "fp64")
    ctx.m2m_step(4000)
    w = ctx.state()["w"]
    ctx.m2m_free()
    got = np.log(w / P.what0)
    # (what is compared with is itself off by a rounding of the ratio and two of the logarithm)
    assert np.abs(got + P.entropy_const).max() <= 2.0 ** -53 / k + 6 * 2.0 ** -53
