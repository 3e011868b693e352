"""The FP64 pass: values a step leaves for the next step of the same call,
its division and square root, its cells on bit patterns, its histogram copies."""
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
    Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
    P.Y, P.sigma = Y, Y * 0.5
    P.eps = 0.05 / n
    if P.prior.kind != "flat":
        P.prior = I.PriorSpec(P.prior.kind, 16, 8, 5, P.prior.hernquist)
    return P


def _state(ctx):
    y, D, Dt = ctx.m2m_get_obs()
    return dict(ctx.state(), y=y, Dt=Dt)


# one call of 7 steps (kept values from the second on, through a prior
# recompute) against 7 calls of one step (none kept).  Positions come from the
# same operations; weights differ by the rounding of ln(w/w_hat) carried along
# (2^-53 of it per step, times mu eps dt in the weight) and of sums whose order
# is free: 1e-13 of each value's scale covers both.
@pytest.mark.parametrize("name", ["plain-fp64", "moving-priors", "flat-log", "ifu-lut", "sh-selfcons", "sh-tri",
                                  "sh-full"])
@pytest.mark.parametrize("n", [1, 31, 33, 4097])
def test_one_call_equals_single_steps(name, n):
    P = _problem(name, n)
    a, b = B.from_problem(P, "fp64"), B.from_problem(P, "fp64")
    a.m2m_step(7)
    for _ in range(7):
        b.m2m_step(1)
    ga, gb = _state(a), _state(b)
    exact = not name.startswith("sh-")
    for k in ga:
        if exact and k in ("x", "y", "z", "vx", "vy", "vz") and k != "y":
            np.testing.assert_array_equal(ga[k], gb[k], err_msg=k)
        np.testing.assert_allclose(ga[k], gb[k], rtol=1e-12 if exact else 1e-9,
                                   atol=1e-13 * np.abs(gb[k]).max(), err_msg=k)
    a.m2m_free()
    b.m2m_free()


# a caller may rescale its weights and move its particles between calls
def test_nothing_is_kept_between_calls():
    P = _problem("moving-priors", 4097)
    a = B.from_problem(P, "fp64")
    a.m2m_step(3)
    a.t["w"].mul_(1.25)
    a.t["x"].neg_()
    a.t["vx"].neg_()
    torch.cuda.synchronize()
    g0 = {k: v.clone() for k, v in a.t.items()}
    _, _, Dt = a.m2m_get_obs()
    a.m2m_step(1)
    x, v = np.stack([g0[k].cpu().numpy() for k in "xyz"]), np.stack([g0[k].cpu().numpy() for k in ("vx", "vy", "vz")])
    want = O.kdk(*x, *v, P.potential, P.dt)
    got = a.state()
    for k, q in zip(("x", "y", "z", "vx", "vy", "vz"), want):
        np.testing.assert_array_equal(got[k], q, err_msg=k)
    w, what = g0["w"].cpu().numpy(), g0["what"].cpu().numpy()
    y = O.observe(*want, w, P.obs, P.incl_sin, P.incl_cos)
    D = (y - P.Y) / P.sigma
    Dt = P.alpha * D + (1 - P.alpha) * Dt
    kern = O.cells_and_kernels(*want, P.obs, P.incl_sin, P.incl_cos)
    dot = O.kernel_dot(kern, Dt / P.sigma, P.obs, P.n)
    np.testing.assert_allclose(got["w"], O.update_weights(w, what, dot, P.eps, P.mu, P.dt), rtol=1e-13)


# the correctly rounded quotient and root at every magnitude they take a
# different route at (the exponent range of the short form, its edges, zeros)
@pytest.mark.parametrize("comps", [[I.PotentialComponent("hernquist", (1.7, 0.3))],
                                   [I.PotentialComponent("log", (0.9, 0.11, 0.77))]])
def test_push_is_bit_exact_at_every_magnitude(comps):
    rng = np.random.default_rng(5)
    n = 200_000
    mag = 2.0 ** rng.uniform(-170, 170, n)
    mag[:1000] = 2.0 ** rng.uniform(-400, -240, 1000)
    mag[1000:2000] = 2.0 ** rng.uniform(240, 330, 1000)
    pos = rng.normal(size=(3, n)) * mag
    pos[:, 2000:2003] = 0.0
    pos[:, 2003:60_000] = rng.normal(size=(3, 57_997))
    vel = rng.normal(size=(3, n))
    P = _problem("plain-fp64", n)
    P.pos, P.vel, P.potential = pos, vel, comps
    ctx = B.from_problem(P, "fp64")
    ctx.m2m_push(1)
    g = ctx.state()
    with np.errstate(all="ignore"):
        want = O.kdk(*pos, *vel, comps, P.dt)
    for k, q in zip(("x", "y", "z", "vx", "vy", "vz"), want):
        np.testing.assert_array_equal(g[k], q, err_msg=k)


# cells at edges, zeros of both signs, NaN and infinities, decided on the bits
def test_cells_at_edges_zeros_and_non_finite_values():
    e = I.uniform_edges(8, -2.0, 2.0)
    V, S = np.zeros(16), np.ones(16)
    vals = np.concatenate([e, np.nextafter(e, -9), np.nextafter(e, 9), [0.0, -0.0, np.nan, -np.nan, np.inf, -np.inf,
                                                                     5e-324, -5e-324, 1e-300, -1e-300, 3.0, -3.0]])
    xs, ys = (q.ravel() for q in np.meshgrid(vals, vals))
    n = xs.size
    P = _problem("flat-log", n)
    P.obs = [I.ObservableSet("grid", "mass", e, e.copy()),
             I.ObservableSet("grid", "gh", e[::2].copy(), e[::2].copy(), gh_V=V, gh_S=S, sigma_kernel=0.1)]
    P.pos = np.stack([xs, -ys, np.zeros(n)])      # Y = z sin i - y cos i with i = 0
    P.incl_sin, P.incl_cos = 0.0, 1.0
    P.vel = np.zeros((3, n))
    P.Y = P.sigma = None
    ctx = B.from_problem(P, "fp64", targets=False)
    ctx.m2m_observe(0)
    y, _, _ = ctx.m2m_get_obs()
    ctx.m2m_set_layout(0)
    ctx.m2m_observe(0)
    walk, _, _ = ctx.m2m_get_obs()
    X, Y = P.pos[0], P.pos[2] * 0.0 - P.pos[1] * 1.0
    want = np.zeros(64)
    with np.errstate(invalid="ignore"):
        for c in range(64):
            i, j = c % 8, c // 8
            ok = (X >= e[i]) & (X < e[i + 1]) & (Y >= e[j]) & (Y < e[j + 1])
            want[c] = P.w0[ok].sum()
    np.testing.assert_allclose(y[:64], want, rtol=n * 2.0 ** -53)
    np.testing.assert_allclose(walk, y, rtol=n * 2.0 ** -53, atol=n * 2.0 ** -53 * want.sum())
