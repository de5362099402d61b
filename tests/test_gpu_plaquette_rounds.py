"""The mean plaquette where a block takes several items (one round, two, three,
and an item cut short by the time extent), against the kernel of
su2_plaquette_noalloc, which has one site per thread."""
import pytest

from paper_1010_1486_gb300 import su2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ns,nt", [(2, 2), (2, 1000), (4, 6), (20, 20), (24, 22), (34, 10), (40, 40), (44, 18), (50, 14),
                                   (54, 20), (64, 10), (100, 2)])
def test_plaquette_of_any_number_of_rounds(ns, nt):
    torch = pytest.importorskip("torch")
    h = su2.su2_create(ns, nt, 2.3, ns + nt, su2.SU2_HOT)
    try:
        su2.su2_set_sampler(h, su2.SU2_SAMPLER_KP)
        su2.su2_heatbath_sweep(h, 1)
        got = su2.su2_plaquette(h)
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        su2.su2_plaquette_noalloc(su2.su2_device_links(h)[0], ns, nt, out.data_ptr(), None)
        torch.cuda.synchronize()
        # six products of binary32 per site, each within 2e-6 of the exact one; the same ones here and there but for
        # the order of the sums
        assert abs(got - out.item()) <= 6 * 2.0 ** -24
        assert su2.su2_plaquette(h) == got
    finally:
        su2.su2_destroy(h)
