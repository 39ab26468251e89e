"""The one-launch forms that run a sample in one CTA or cluster, at the sizes
where their splits change: bit for bit against the oracle."""
import numpy as np
import pytest

from test_gpu_rec import _built, assert_same, dev, oracle_run, snn, workload  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B,NI,N,NO,T", [
    (1, 40, 1100, 10, 40),     # clusters of four CTAs, the last with a short column range
    (2, 1030, 64, 40, 40),     # more outputs than lanes, two warps of neurons, ragged input words
    (153, 33, 520, 3, 20),     # one CTA per sample, more samples than SMs
    (2, 64, 4200, 10, 12),     # clusters of eight
    (80, 24, 4200, 10, 6),     # two CTAs by the layer's width, eight neurons per thread
])
def test_rec_gather_one_launch(B, NI, N, NO, T):
    """Two runs, the second continuing, and the tensor form's operands left so
    that a per-step (profiled) run continues too."""
    p, r, s, wf, wr, wo = workload(B, NI, N, NO, seed=B)
    net = snn().RecNetwork(p, wf, wr, wo)
    st, rh, ri = oracle_run(p, r, s, wf, wr, wo, T)
    assert rh.sum() > 0
    net.run(dev(r), dev(s), T, record=True, record_input=True, form="gather")
    assert_same(net, st, rh, ri)
    for profile in (False, True):
        st, rh, ri = oracle_run(p, r, s, wf, wr, wo, 3, st=st, episodic=False)
        net.run(dev(r), dev(s), 3, continue_=True, record=True, record_input=True, form="gather", profile=profile)
        assert_same(net, st, rh, ri)
    net.close()
