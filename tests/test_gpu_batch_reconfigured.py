"""A batch whose models are reconfigured through their contexts: flush form,
potential, layout, against separate contexts given the same calls."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


def _log(q):
    q.m2m_potential([I.PotentialComponent("log", (0.9, 0.2, 0.8))])


def _same_kind(q):
    q.m2m_potential([I.PotentialComponent("hernquist", (1.3, 0.7)), I.PotentialComponent("nfw", (0.01, 7.0))])


def _sh(q):
    q.m2m_potential([I.PotentialComponent("sh", (32, 0.01, 50.0, 2))])


# what is called, on which models, and whether the next batch step is fused;
# every state and observable bit for bit
@pytest.mark.parametrize("what,which,fused", [
    (lambda q: q.m2m_set_pipeline(2), (1,), 2), (lambda q: q.m2m_set_pipeline(2), (0, 1, 2), 2),
    (_log, (1,), 2), (_log, (0, 1, 2), 2), (_same_kind, (0, 2), 2), (_sh, (2,), 0),
    (lambda q: q.m2m_set_layout(0), (1,), 0), (lambda q: q.m2m_set_layout(0), (0, 1, 2), 0)])
def test_reconfigured_models_step_as_by_themselves(what, which, fused):
    from paper_1207_6403_gb300 import m2m
    probs = []
    for m, n in enumerate((5000, 33, 20_001)):
        P = I.make_scan([(I.HALO_MASS_RATIOS[m], I.HALO_RS[m])], (2.0, 5.0), n=n, n_target=50)[0]
        rng = np.random.default_rng(m)
        P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
        P.sigma = P.Y * 0.5
        P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
        P.eps = 0.05 / 1_000_000
        probs.append(P)
    b = m2m.m2m_batch_init("fp32c", probs)
    own = [b.m2m_batch_context(m) for m in range(3)]
    alone = [m2m.from_problem(P, "fp32c") for P in probs]

    def step(n, mode):
        b.m2m_batch_step(n)
        assert b.m2m_batch_fused() == mode
        for m, (q, c) in enumerate(zip(own, alone)):
            c.m2m_step(n)
            g, want = q.state(), c.state()
            for k in want:
                np.testing.assert_array_equal(g[k], want[k], err_msg=f"model {m} {k}")
            for u, v in zip(q.m2m_get_obs(), c.m2m_get_obs()):
                np.testing.assert_array_equal(u, v, err_msg=f"model {m}")

    step(4, 2)
    for m in which:
        what(own[m])
        what(alone[m])
    step(4, fused)
    step(4, fused)
    b.m2m_batch_free()
    for c in alone:
        c.m2m_free()
