"""The fused batch's segments: models of very different size, several models
in one block and one model over many, calls of odd and even step counts (the
record of a step is written by the pass that follows)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("sizes", [[1], [1, 31, 1023, 5000, 70_001], [300_007, 33], [257] * 40])
def test_segments_equal_single_models(sizes, moving):
    from paper_1207_6403_gb300 import m2m
    halos = [(I.HALO_MASS_RATIOS[m % 6], I.HALO_RS[m % 8]) for m in range(len(sizes))]
    probs = []
    for m, n in enumerate(sizes):
        P = I.make_scan([halos[m]], (2.0, 5.0), n=n, n_target=50)[0]
        rng = np.random.default_rng(m)
        P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
        P.sigma = P.Y * 0.5
        P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
        P.eps = 0.05 / 1_000_000          # (0.05/31 lets the weights of 31 particles run off to zero)
        if moving:
            P.prior = I.PriorSpec("e_lz", 8, 8, 3)
        probs.append(P)
    b = m2m.m2m_batch_init("fp32c", probs)
    alone = [m2m.from_problem(P, "fp32c") for P in probs]
    for steps in (1, 2, 5, 2):
        b.m2m_batch_step(steps)
        assert b.m2m_batch_fused() == 2
        recs = b.m2m_batch_get_records()
        for m, c in enumerate(alone):
            c.m2m_step(steps)
            q = b.m2m_batch_context(m)
            g, want = q.state(), c.state()
            for k in want:
                np.testing.assert_array_equal(g[k], want[k], err_msg=f"model {m} {k}")
            for u, v in zip(q.m2m_get_obs(), c.m2m_get_obs()):
                np.testing.assert_array_equal(u, v)
            r = c.m2m_get_record()
            assert recs[m]["step"] == r["step"] and recs[m]["chi2"] == pytest.approx(r["chi2"], rel=1e-12)
            # float partials grouped differently
            assert recs[m]["sum_w"] == pytest.approx(r["sum_w"], rel=1e-5)
            assert recs[m]["S"] == pytest.approx(r["S"], rel=1e-4, abs=1e-6)
    # a model of the batch stepped alone, then the batch again
    q = b.m2m_batch_context(0)
    q.m2m_step(1)
    alone[0].m2m_step(1)
    assert q.m2m_get_record()["step"] == alone[0].m2m_get_record()["step"]
    np.testing.assert_array_equal(q.state()["w"], alone[0].state()["w"])
