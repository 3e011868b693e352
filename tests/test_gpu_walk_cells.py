"""The FP32C run-time set walk: cells kept from the scatter for the update,
sets that share their edges, the branch-free bisection, against the oracle."""
import numpy as np
import pytest

from oracle import m2m as O
from paper_1207_6403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1207_6403_gb300 import m2m as B  # noqa: E402


def _sets(kind):
    S, e = I.ObservableSet, lambda nb: np.cumsum(np.concatenate([[0.01], np.linspace(0.02, 0.5, nb)]))
    sk = 0.1
    if kind == "shared":            # two annulus sets with equal edges, one with others, GH apertures
        g = np.array([-3.0, -1.0, -0.4, 0.0, 0.7, 2.5])
        return [S("annulus", "mass", e(37)), S("annulus", "vlos2", e(37)), S("annulus", "mass", e(36)),
                S("grid", "gh", g, g.copy(), gh_V=np.full(25, 0.1), gh_S=np.full(25, 0.5), sigma_kernel=sk)]
    if kind == "wide":              # 13 + 13 + 13 bits: the cells do not fit the packed word
        return [S("shell", "mass", e(1100)), S("annulus", "mass", e(2100)), S("annulus", "vlos2", e(2101))]
    if kind == "one":               # one cell per set
        return [S("shell", "mass", np.array([0.0, 1.3])), S("annulus", "gh", np.array([0.1, 2.0]), gh_V=np.zeros(1),
                                                            gh_S=np.ones(1), sigma_kernel=sk)]
    u = I.uniform_edges(6, -1.0, 1.0)
    return [S("grid", "vlos2", u, u.copy()), S("grid", "gh", u, u.copy(), gh_V=np.zeros(36), gh_S=np.ones(36),
                                               sigma_kernel=sk, psf_q=I.gaussian_psf_table(0.2, 6), psf_seed=9),
            S("grid", "mass", u, u.copy())]


# the weights after 6 steps, every one (FP32C's 1e-4 after 1000 steps; one
# step's update is held to 2e-7 elsewhere, so 6 of them to 2e-6), and the
# observables to 1e-5 of their largest
@pytest.mark.parametrize("kind", ["shared", "wide", "one", "seeing"])
@pytest.mark.parametrize("n", [1, 33, 20_001])
def test_walk_matches_the_oracle(kind, n):
    P = I.make_problem("plain-fp64", n=n, precision="fp32c", with_target=False)
    P.obs = _sets(kind)
    rng = np.random.default_rng(n)
    P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
    P.w0[::50] *= 150.0             # past the fast range of the fixed-point histogram
    P.eps = 1e-8
    P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
    P.sigma = P.Y * 0.5
    ctx = B.from_problem(P, "fp32c")
    for steps in (1, 3, 2):
        ctx.m2m_step(steps)
    g = ctx.state()
    y, _, _ = ctx.m2m_get_obs()
    st = O.run(P, 6, precision="fp32c")
    np.testing.assert_array_equal(g["x"], st.x)
    np.testing.assert_allclose(g["w"], st.w, rtol=2e-6)
    np.testing.assert_allclose(y, st.y_obs, rtol=0, atol=1e-5 * np.abs(st.y_obs).max())
    # a caller that moves the particles observes before it updates
    ctx.t["x"].neg_()
    torch.cuda.synchronize()
    ctx.m2m_observe(0)
    ctx.m2m_update_weights()
    ctx.m2m_free()


# a velocity that gives no finite moment is reported, not dropped
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e25])
@pytest.mark.parametrize("weight", [0.0, 1.0])
def test_walk_reports_moments_that_are_not_finite(bad, weight):
    n = 100
    P = I.make_problem("plain-fp64", n=n, precision="fp32c", with_target=False)
    P.obs = _sets("shared")[3:]
    P.pos[:, 7] = (0.1, 0.1, 0.0)
    P.vel[:, 7] = bad
    P.w0[7] *= weight
    with pytest.raises(B.M2MError):
        B.from_problem(P, "fp32c", targets=False)
