"""Small lattices run whole calls in one launch (a thread-block cluster); with
su2_set_timing on they run phase by phase.  Both are the same chain: links and
trial counts bit for bit, at the edges of the cluster's split (less than a
warp, ragged CTAs, one to sixteen CTAs, with and without warps that draw
ahead, the largest small lattice and the first that is not), with
over-relaxation, reunitarization, sparse measurements, low trial caps and more
sweeps than one launch takes.  The binary64 sums differ in order only."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu

KP, CREUTZ = su2.SU2_SAMPLER_KP, su2.SU2_SAMPLER_CREUTZ


def _run(ns, nt, beta, sampler, timing, calls, overrelax=0, cap=None, start=su2.SU2_HOT):
    h = su2.su2_create(ns, nt, beta, 77, start)
    out = []
    try:
        su2.su2_set_sampler(h, sampler)
        su2.su2_set_overrelax(h, overrelax)
        su2.su2_set_timing(h, timing)
        if cap:
            su2.su2_set_trial_cap(h, cap)
        for nsweeps, every, reunit in calls:
            try:
                plaq, poly, stats = su2.su2_generate(h, nsweeps, every, reunit)
                out.append((plaq, poly, stats["trials"], 0))
            except su2.SU2Error as e:
                out.append((None, None, None, e.status))
        su2.su2_heatbath_sweep(h, 2)
        return out, su2.su2_get_links(h, ns, nt), su2.su2_get_state(h)["sweep"]
    finally:
        su2.su2_destroy(h)


def _same(ns, nt, beta, sampler, calls, **kw):
    (a, links_a, sweep_a), (b, links_b, sweep_b) = (_run(ns, nt, beta, sampler, t, calls, **kw) for t in (False, True))
    assert sweep_a == sweep_b
    assert np.array_equal(links_a, links_b)
    for (pa, la, ta, sa), (pb, lb, tb, sb) in zip(a, b):
        assert sa == sb and ta == tb
        if pa is not None:
            # sums of at most 6 V terms of order one, in another order
            tol = 8 * ns ** 3 * nt * 2.0 ** -53
            assert np.allclose(pa, pb, rtol=0, atol=tol) and np.allclose(la, lb, rtol=0, atol=tol)


@pytest.mark.parametrize("ns,nt", [(2, 2), (2, 6), (4, 4), (6, 4), (6, 6), (8, 8), (10, 2), (8, 18), (12, 8), (16, 4),
                                   (20, 2), (16, 6)])
@pytest.mark.parametrize("sampler", [KP, CREUTZ])
def test_every_split(ns, nt, sampler):
    _same(ns, nt, 2.3, sampler, [(3, 1, 0), (2, 2, 0)])


@pytest.mark.parametrize("sampler,beta,overrelax", [(KP, 2.3, 1), (KP, 6.0, 3), (CREUTZ, 2.3, 2), (KP, 0.4, 0), (KP, 0.0, 1),
                                                    (CREUTZ, 0.0, 0), (CREUTZ, 20.0, 0), (KP, 1e13, 0)])
def test_options(sampler, beta, overrelax):
    _same(8, 6, beta, sampler, [(5, 2, 0), (4, 1, 2), (3, 3, 1), (2, 0, 1)], overrelax=overrelax)
    _same(6, 12, beta, sampler, [(4, 1, 3)], overrelax=overrelax, start=su2.SU2_COLD)


@pytest.mark.parametrize("sampler,cap", [(KP, 2), (KP, 4), (CREUTZ, 2), (CREUTZ, 6)])
def test_trial_caps(sampler, cap):
    _same(8, 8, 3.0, sampler, [(2, 1, 0), (1, 1, 0)], cap=cap)


def test_more_sweeps_than_one_launch():
    _same(4, 4, 2.3, KP, [(600, 7, 50)])
