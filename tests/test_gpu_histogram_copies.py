"""The FP32C block histogram kept in lane copies (shells + annuli layouts,
1024-thread passes) against the 512-thread passes, which keep one histogram:
exact integer sums, so the state and the observables are equal bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


def _run(P, threads, persistent):
    from paper_1207_6403_gb300 import m2m
    ctx = m2m.from_problem(P, "fp32c")
    ctx.m2m_set_launch(threads)
    ctx.m2m_set_persistent(persistent)
    ctx.m2m_step(3)
    y, D, Dt = ctx.m2m_get_obs()
    out = dict(ctx.state(), y=y, Dt=Dt)
    ctx.m2m_free()
    return out


# 8 copies (short passes), 32 (long ones: 1.3M particles, and again across the
# flush that keeps the part-sums exact), fewer where many bins leave no room
# (1, 2 and 4), with ragged counts of particles and bins
@pytest.mark.parametrize("name,n,shells,annuli", [
    ("moving-priors", 1, 100, 60), ("moving-priors", 4099, 101, 61), ("moving-priors", 1_300_003, 100, 60),
    ("moving-priors", 5_300_001, 97, 3), ("moving-priors", 30_001, 1500, 300), ("moving-priors", 30_001, 1200, 901),
    ("moving-priors", 30_001, 2000, 601), ("plain-fp64", 20_011, 37, 19)])
def test_copies_equal_one_histogram(name, n, shells, annuli):
    P = I.make_problem(name, n=n, precision="fp32c", with_target=False)
    P.obs[0] = I.ObservableSet("shell", "mass", I.log_shell_edges(shells, 0.05, 20.0))
    if name == "plain-fp64":
        e = I.log_shell_edges(annuli, 0.05, 20.0)
        P.obs[1:] = [I.ObservableSet("annulus", "mass", e), I.ObservableSet("annulus", "vlos2", e.copy())]
    else:
        P.obs[1] = I._gh_set_annuli(annuli, 0.05, 20.0, 0.1)
    # weights of very different size: some terms take the histogram's general path
    w = P.w0 * (1.0 + 199.0 * (np.arange(n) % 97 == 5))
    P.w0[:] = w
    rng = np.random.default_rng(3)
    Y = np.abs(rng.normal(size=P.nobs)) + 0.1
    P.Y, P.sigma = Y, Y * 10.0
    want = _run(P, 512, False)
    for persistent in (True, False):
        got = _run(P, 1024, persistent)
        for k in want:
            np.testing.assert_array_equal(got[k], want[k], err_msg=k)
