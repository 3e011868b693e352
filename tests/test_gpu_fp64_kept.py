"""What an FP64 step leaves for the next one of the same call: given back on
request, and the same run with and without it; the pass at the sizes where it
takes 512 threads and two to 32 copies of the histogram."""
import numpy as np
import pytest

from oracle import m2m as O
from paper_1207_6403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1207_6403_gb300 import m2m as B  # noqa: E402


def _problem(name, n):
    P = I.make_problem(name, n=n, precision="fp64", with_target=False)
    rng = np.random.default_rng(n)
    P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
    P.eps = 0.05 / n
    return P


def _targets(P):
    Y = np.abs(np.random.default_rng(7).normal(size=P.nobs)) / P.nobs + 1e-3
    P.Y, P.sigma = Y, Y * 0.5
    return P


# one call of 7 steps with the buffer and without it.  The force and the
# Gauss-Hermite factors are the same functions of the same arguments; the
# logarithm differs by its rounding and the sums by their order: the bounds of
# the same comparison between one call and single steps.
@pytest.mark.parametrize("name", ["plain-fp64", "moving-priors", "flat-log", "ifu-lut", "sh-selfcons", "sh-tri"])
@pytest.mark.parametrize("n", [33, 4097, 100_003])
def test_kept_and_computed_values_agree(name, n):
    P = _targets(_problem(name, n))
    if P.prior.kind != "flat":
        P.prior = I.PriorSpec(P.prior.kind, 16, 8, 5, P.prior.hernquist)
    out = []
    for on in (True, False):
        ctx = B.from_problem(P, "fp64")
        ctx.m2m_set_force_cache(on)
        ctx.m2m_step(7)
        y, _, Dt = ctx.m2m_get_obs()
        out.append(dict(ctx.state(), y_obs=y, Dt=Dt))
        ctx.m2m_free()
    exact = not name.startswith("sh-")
    for k, want in out[0].items():
        if exact and k in ("x", "y", "z", "vx", "vy", "vz"):
            np.testing.assert_array_equal(out[1][k], want, err_msg=k)
        np.testing.assert_allclose(out[1][k], want, rtol=1e-12 if exact else 1e-9, atol=1e-13 * np.abs(want).max(),
                                   err_msg=k)


def test_memory_is_given_back_and_taken_again():
    n = 2_000_000
    ctx = B.from_problem(_targets(_problem("plain-fp64", n)), "fp64")
    for on in (True, False, True):                       # every kernel loaded
        ctx.m2m_set_force_cache(on)
        ctx.m2m_step(2)
    torch.cuda.synchronize()
    free = [torch.cuda.mem_get_info()[0]]
    for on in (False, True, True, False):
        ctx.m2m_set_force_cache(on)
        free.append(torch.cuda.mem_get_info()[0])
        ctx.m2m_step(2)
    ctx.m2m_free()
    assert free[1] - free[0] >= 48 * n                   # (whole pages)
    assert free[1] - free[2] >= 48 * n and free[3] == free[2] and free[4] == free[1]


# (histogram copies that the rule gives on 152 SMs: 32, 16, 8, 4, 2 of
# 5-moment and of single cells; 512 threads from 77,824 particles on, 256
# below, where fewer particles give fewer copies), 3 steps against the oracle.
# Each y_j is a sum of n terms in a free order (n 2^-53 of the sum of the
# weights, sqrt 2 or v^2 of it for the moments); its part in the weights is
# smaller by eps dt alpha / sigma^2, below 1e-13 here.
@pytest.mark.parametrize("n", [40_001, 100_003])
@pytest.mark.parametrize("name,shells,annuli", [
    ("moving-priors", 5, 3), ("moving-priors", 21, 11), ("moving-priors", 97, 41), ("moving-priors", 150, 81),
    ("moving-priors", 301, 141), ("plain-fp64", 3, 2), ("plain-fp64", 37, 19), ("plain-fp64", 101, 200),
    ("flat-log", 4, 2), ("flat-log", 12, 6), ("ifu-lut", 0, 0)])
def test_large_passes_match_the_oracle(name, shells, annuli, n):
    P = _problem(name, n)
    P.prior = I.PriorSpec("flat")
    if name == "moving-priors":
        P.obs = [I.ObservableSet("shell", "mass", I.log_shell_edges(shells, 0.05, 20.0)),
                 I._gh_set_annuli(annuli, 0.05, 20.0, 0.1)]
    elif name == "plain-fp64":
        e = I.log_shell_edges(annuli, 0.05, 20.0)
        P.obs = [I.ObservableSet("shell", "mass", I.log_shell_edges(shells, 0.05, 20.0)),
                 I.ObservableSet("annulus", "mass", e), I.ObservableSet("annulus", "vlos2", e.copy())]
    elif name == "flat-log":
        g, h = I.uniform_edges(shells, -1.0, 1.0), I.uniform_edges(annuli, -1.0, 1.0)
        c = annuli * annuli
        P.obs = [I.ObservableSet("grid", "mass", g, g.copy()),
                 I.ObservableSet("grid", "gh", h, h.copy(), gh_V=np.full(c, 0.1), gh_S=np.full(c, 0.6),
                                 sigma_kernel=0.1)]
    _targets(P)
    ctx = B.from_problem(P, "fp64")
    ctx.m2m_step(3)
    got = ctx.state()
    y, _, _ = ctx.m2m_get_obs()
    ctx.m2m_free()
    st = O.run(P, 3, precision="fp64")
    for k in ("x", "y", "z", "vx", "vy", "vz"):
        np.testing.assert_array_equal(got[k], getattr(st, k), err_msg=k)
    big = max(2.0, float((np.abs(P.vel).max() ** 2) * 3)) if name == "plain-fp64" else 2.0
    np.testing.assert_allclose(y, st.y_obs, rtol=0, atol=n * 2.0 ** -53 * big * P.w0.sum())
    np.testing.assert_allclose(got["w"], st.w, rtol=1e-12)
