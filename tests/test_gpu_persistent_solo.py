"""The persistent kernel's solo residual (at most 512 observables, launches of
three steps or more) against separate launches, around both limits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


@pytest.mark.parametrize("shells,annuli", [(1, 1), (7, 2), (100, 60), (12, 100), (13, 100)])
@pytest.mark.parametrize("n", [1, 4097, 200_003])
def test_solo_equals_separate_launches(shells, annuli, n):
    from paper_1207_6403_gb300 import m2m
    P = I.make_problem("moving-priors", n=n, precision="fp32c", with_target=False)
    P.obs[0] = I.ObservableSet("shell", "mass", I.log_shell_edges(shells, 0.05, 20.0))
    P.obs[1] = I._gh_set_annuli(annuli, 0.05, 20.0, 0.1)
    P.prior = I.PriorSpec("e_lc", 16, 8, 9, (1.0, 1.0))
    rng = np.random.default_rng(n)
    P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
    P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
    P.sigma = P.Y * 0.5
    P.sigma[::7] = 0.0                   # masked
    got = []
    for persistent in (True, False):
        ctx = m2m.from_problem(P, "fp32c")
        ctx.m2m_set_persistent(persistent)
        out = []
        for steps in (1, 2, 3, 4, 11, 5):            # launches of 1 to 8 steps, priors due at 9 and 18
            ctx.m2m_step(steps)
            out.append((ctx.state(), ctx.m2m_get_obs(), ctx.m2m_get_record()))
        out.append(ctx.m2m_get_history(1, 26))
        ctx.m2m_free()
        got.append(out)
    for (s0, o0, r0), (s1, o1, r1) in zip(got[0][:-1], got[1][:-1]):
        for k in s0:
            np.testing.assert_array_equal(s0[k], s1[k], err_msg=k)
        for u, v in zip(o0, o1):
            np.testing.assert_array_equal(u, v)
    for a, b in zip(got[0][-1], got[1][-1]):
        assert a["step"] == b["step"]
        for k in ("chi2", "chi2_raw", "max_abs_dt"):
            assert a[k] == pytest.approx(b[k], rel=1e-12)
        assert a["sum_w"] == pytest.approx(b["sum_w"], rel=1e-5)
        assert a["S"] == pytest.approx(b["S"], rel=1e-4, abs=1e-6)
