"""A fused batch between steps of its models by themselves: the arguments and
the step counter that the batch keeps on the device, the record tickets, the
graphs captured before, against separate contexts."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

I = pytest.importorskip("paper_1207_6403_gb300.inputs")


# 3 steps of every model alone (odd), then 2 (even), an observe, a lazy update
# left pending and applied, another launch shape (no histogram copies: another
# shared memory size), each followed by batch calls of step counts whose graphs
# exist already.  State and observables bit for bit; the records' S and sum of
# weights are float partials grouped differently.
@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("sizes", [[1, 1023, 5000], [70_001, 33, 40_000, 257]])
def test_batch_after_its_models_moved_on(sizes, moving):
    from paper_1207_6403_gb300 import m2m
    probs = []
    for m, n in enumerate(sizes):
        P = I.make_scan([(I.HALO_MASS_RATIOS[m % 6], I.HALO_RS[m % 8])], (2.0, 5.0), n=n, n_target=50)[0]
        rng = np.random.default_rng(m)
        P.Y = np.abs(rng.normal(size=P.nobs)) / P.nobs + 1e-3
        P.sigma = P.Y * 0.5
        P.w0[:] = np.exp(0.3 * rng.normal(size=n)) / n
        P.eps = 0.05 / 1_000_000
        if moving:
            P.prior = I.PriorSpec("e_lz", 8, 8, 3)
        probs.append(P)
    b = m2m.m2m_batch_init("fp32c", probs)
    own = [b.m2m_batch_context(m) for m in range(len(sizes))]
    alone = [m2m.from_problem(P, "fp32c") for P in probs]

    def both(f):
        for q, c in zip(own, alone):
            f(q)
            f(c)

    def batch(steps):
        b.m2m_batch_step(steps)
        assert b.m2m_batch_fused() == 2
        recs = b.m2m_batch_get_records()
        for m, c in enumerate(alone):
            c.m2m_step(steps)
            r = c.m2m_get_record()
            assert recs[m]["step"] == r["step"] and recs[m]["chi2"] == pytest.approx(r["chi2"], rel=1e-12)
            assert recs[m]["sum_w"] == pytest.approx(r["sum_w"], rel=1e-5)
            assert recs[m]["S"] == pytest.approx(r["S"], rel=1e-4, abs=1e-6)

    def same(what):
        for m, (q, c) in enumerate(zip(own, alone)):
            g, want = q.state(), c.state()
            for k in want:
                np.testing.assert_array_equal(g[k], want[k], err_msg=f"{what}: model {m} {k}")
            for u, v in zip(q.m2m_get_obs(), c.m2m_get_obs()):
                np.testing.assert_array_equal(u, v, err_msg=f"{what}: model {m}")
            assert q.m2m_get_record()["step"] == c.m2m_get_record()["step"], what

    def lazy(q):
        q.m2m_set_lazy_update(True)
        q.m2m_step(1)
        q.m2m_finish_update()
        q.m2m_set_lazy_update(False)

    for steps in (1, 2, 5):                       # captured
        batch(steps)
    same("batch")
    for what, f in (("3 alone", lambda q: q.m2m_step(3)), ("2 alone", lambda q: q.m2m_step(2)),
                    ("observed", lambda q: q.m2m_observe(0)), ("lazy", lazy),
                    ("512 threads", lambda q: (q.m2m_set_launch(512), q.m2m_step(1))),
                    ("1024 threads", lambda q: q.m2m_set_launch(1024))):
        both(f)
        same(what)
        for steps in (2, 5, 1):
            batch(steps)
        same(what + ", then the batch")
    # one model alone in another shape
    for q in (own[0], alone[0]):
        q.m2m_set_launch(256)
    batch(2)
    same("one model with 256 threads")
    b.m2m_batch_free()
    for c in alone:
        c.m2m_free()
