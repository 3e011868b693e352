"""The FP32C run-time set walk after its caller moved the particles: the update
takes the cells that the observe between left, not those of the old places."""
import numpy as np
import pytest

from oracle import m2m as O
from paper_1207_6403_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1207_6403_gb300 import m2m as B  # noqa: E402
from test_gpu_walk_cells import _sets  # noqa: E402


# positions scaled by 0.6 and turned, so that most particles change their cell
# in every set.  One update: 2e-7 of the weight (the bound of a step elsewhere)
# and 2e-6 of its change (some thirty float roundings of the sum over the sets)
@pytest.mark.parametrize("kind", ["shared", "wide", "one", "seeing"])
@pytest.mark.parametrize("n", [33, 20_001])
def test_update_after_the_particles_were_moved(kind, n):
    P = I.make_problem("plain-fp64", n=n, precision="fp32c", with_target=False)
    P.obs = _sets(kind)
    rng = np.random.default_rng(n)
    P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
    P.alpha = 1.0
    P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
    P.sigma = P.Y * 0.5
    # an adaptation rate that moves the fastest weight by a hundredth a step
    pv = [np.asarray(q, np.float32) for q in (*P.pos, *P.vel)]
    kern = O.cells_and_kernels(*pv, P.obs, P.incl_sin, P.incl_cos)
    coef = (O.observe_from(kern, P.w0, P.obs) - P.Y) / P.sigma ** 2
    P.eps = 0.01 / (P.dt * np.abs(O.kernel_dot(kern, coef, P.obs, n)).max())
    ctx = B.from_problem(P, "fp32c")
    ctx.m2m_step(2)
    t = ctx.t
    x, y = t["x"].clone(), t["y"].clone()
    t["x"].copy_(-0.6 * y)
    t["y"].copy_(0.6 * x)
    t["z"].mul_(0.6)
    torch.cuda.synchronize()
    before = {k: v.clone().cpu().numpy() for k, v in t.items()}
    ctx.m2m_observe(1)
    ctx.m2m_update_weights()
    got = ctx.state()["w"]
    y_got, _, Dt = ctx.m2m_get_obs()
    ctx.m2m_free()
    pv = [before[k] for k in ("x", "y", "z", "vx", "vy", "vz")]
    kern = O.cells_and_kernels(*pv, P.obs, P.incl_sin, P.incl_cos, epoch=2)
    want_y = O.observe(*pv, before["w"], P.obs, P.incl_sin, P.incl_cos, epoch=2)
    np.testing.assert_allclose(y_got, want_y, rtol=0, atol=1e-5 * np.abs(want_y).max())
    dot = O.kernel_dot(kern, Dt / P.sigma, P.obs, n)
    want = O.update_weights(before["w"], before["what"], dot, P.eps, P.mu, P.dt)
    moved = np.abs(np.log(want / before["w"]))
    assert moved.max() > 1e-3                 # the update can be seen
    np.testing.assert_allclose(got, want, rtol=2e-7 + 2e-6 * moved.max())
