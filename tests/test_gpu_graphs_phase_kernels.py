"""The captured generation graphs, on lattices of more than 8,192 links per
phase (smaller ones run whole calls in one launch and capture nothing): replays
against eager launches bit for bit through every measurement and
reunitarization variant, captured again after each setting they depend on."""
import numpy as np
import pytest

from paper_1010_1486_gb300 import su2
from test_gpu_graphs import SCRIPT, run

pytestmark = pytest.mark.gpu
SU2_E_SAMPLER = 4
# sparse measurement with reunitarization on and off the measured sweeps, history growing and not
SPARSE = [("gen", 6, 2, 2), ("gen", 6, 2, 3), ("gen", 6, 3, 2), ("or", 1), ("gen", 6, 2, 3), ("gen", 13, 1, 4),
          ("beta", 2.0), ("gen", 6, 2, 3), ("sampler", su2.SU2_SAMPLER_KP), ("gen", 6, 2, 3), ("state", 7),
          ("gen", 5, 0, 2), ("gen", 40, 1, 0)]


@pytest.mark.parametrize("ns,nt,script", [(14, 14, SCRIPT), (12, 10, SPARSE), (26, 2, SPARSE), (16, 8, SCRIPT)])
def test_graph_replays_equal_eager_launches(ns, nt, script):
    torch = pytest.importorskip("torch")
    assert ns ** 3 * nt // 2 > 8192
    eager = run(None, ns, nt, script)
    graphs = run(torch.cuda.Stream(), ns, nt, script)
    assert len(eager) == len(graphs)
    for a, b in zip(eager[:-2], graphs[:-2]):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
        assert a[2] == b[2] and a[3] == b[3]
    assert np.array_equal(eager[-2], graphs[-2])
    assert eager[-1] == graphs[-1]


@pytest.mark.parametrize("sampler", [su2.SU2_SAMPLER_CREUTZ, su2.SU2_SAMPLER_KP])
def test_trial_cap_change_captures_again(sampler):
    torch = pytest.importorskip("torch")
    # cold at beta = 6: Kennedy-Pendleton needs more than two trials for a few links in a thousand
    h = su2.su2_create(14, 14, 6.0, 7, su2.SU2_COLD, stream=torch.cuda.Stream())
    ref = su2.su2_create(14, 14, 6.0, 7, su2.SU2_COLD)
    try:
        for x in (h, ref):
            su2.su2_set_sampler(x, sampler)
            su2.su2_generate(x, 2, 1, 0)
            su2.su2_set_trial_cap(x, 2)
            with pytest.raises(su2.SU2Error) as err:
                su2.su2_generate(x, 1, 1, 0)
            assert err.value.status == SU2_E_SAMPLER
            su2.su2_set_trial_cap(x, 4096)
            su2.su2_generate(x, 2, 1, 0)
        assert np.array_equal(su2.su2_get_links(h, 14, 14), su2.su2_get_links(ref, 14, 14))
    finally:
        su2.su2_destroy(h)
        su2.su2_destroy(ref)
