"""FP64 cells of radial sets whose squared edges lie below the normal float
range: the index guess is a float, the cells are those of the doubles."""
import numpy as np
import pytest

from oracle import m2m as O
from paper_1207_6403_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# r^2 from 1e-44 up through 2^-126 (1.2e-38) to 1e-34, shells + GH annuli and
# shells + mass and v^2 annuli
@pytest.mark.parametrize("name", ["moving-priors", "plain-fp64"])
@pytest.mark.parametrize("nb", [1, 7, 60])
def test_cells_below_the_float_range(name, nb):
    from paper_1207_6403_gb300 import m2m as B
    rng = np.random.default_rng(nb)
    n = 997
    P = I.make_problem(name, n=n, precision="fp64", with_target=False)
    edges = I.log_shell_edges(nb, 1e-22, 1e-17)
    sk = P.obs[-1].sigma_kernel
    if name == "plain-fp64":
        P.obs = [I.ObservableSet("shell", "mass", edges), I.ObservableSet("annulus", "mass", edges.copy()),
                 I.ObservableSet("annulus", "vlos2", edges.copy())]
    else:
        P.obs = [I.ObservableSet("shell", "mass", edges),
                 I.ObservableSet("annulus", "gh", edges.copy(), gh_V=np.zeros(nb), gh_S=np.ones(nb), sigma_kernel=sk)]
    r = np.exp(rng.uniform(np.log(0.5e-22), np.log(2e-17), n))
    u = rng.normal(size=(3, n))
    P.pos = u / np.sqrt((u * u).sum(0)) * r
    P.w0 = rng.random(n) / n
    P.Y = P.sigma = None
    ctx = B.from_problem(P, "fp64", targets=False)
    ctx.m2m_observe(0)
    y, _, _ = ctx.m2m_get_obs()
    ctx.m2m_free()
    want = O.observe(*P.pos, *P.vel, P.w0, P.obs, P.incl_sin, P.incl_cos)
    # sums of at most n terms in another order; a Gauss-Hermite moment is at most sqrt 2 of the weight
    np.testing.assert_allclose(y, want, rtol=0, atol=n * 2.0 ** -53 * 2.0 * max(1.0, np.abs(P.vel).max() ** 2 * 3))
