"""The fused forms (a sample in one CTA or cluster for a whole run; a step in one
launch over column tiles) at the sizes where their splits change: bit for bit
against the oracle."""
import numpy as np
import pytest

from test_gpu_rec import _built, assert_same, bits, dev, dyadic_workload, oracle_run, snn, workload  # noqa: F401

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


@pytest.mark.parametrize("B,NI,N,NO", [
    (1, 33, 200, 256),         # one item per part, the widest readout, unpaired operand columns
    (300, 64, 700, 40),        # tiles in four parts, the last pair of CTAs with 44 samples in one
    (2200, 40, 700, 10),       # tiles in two parts, ragged in the second
    (2560, 64, 2000, 10),      # a full round and the rest of the tiles in four parts
])
def test_rec_tensor_form_cut_tiles(B, NI, N, NO):
    """Samples of the first CTA, the second CTA and the last one against oracle
    runs of that sample alone (dyadic weights)."""
    T = 12
    p, r, s, wf, wr, wo = dyadic_workload(B, NI, N, NO, seed=N)
    net = snn().RecNetwork(p, wf, wr, wo)
    net.run(dev(r), dev(s), T, record=True, form="tensor")
    got = {name: net.read(name) for name in ("raster", "v", "i_syn", "v_out", "counts")}
    net.close()
    for b in sorted({0, min(B - 1, 131), B - 1}):
        st, rh, _ = oracle_run(p, r[b:b + 1], s[b:b + 1], wf, wr, wo, T)
        assert rh.sum() > 0
        assert np.array_equal(got["raster"][:, b], rh[:, 0]), b
        for name, ref in (("v", st.v), ("i_syn", st.i_syn), ("v_out", st.v_out), ("counts", st.counts)):
            assert np.array_equal(bits(got[name][b]), bits(ref[0])), (b, name)


def test_rec_tensor_form_counts_without_their_ring():
    """A tensor run recorded by a capture, the first of its batch size, may not
    allocate: the counts then take each step's spikes."""
    B, NI, N, NO, T = 130, 64, 300, 10, 40
    p, r, s, wf, wr, wo = dyadic_workload(B, NI, N, NO, seed=3)
    st, rh, _ = oracle_run(p, r, s, wf, wr, wo, T)
    assert rh.sum() > 0
    net = snn().RecNetwork(p, wf, wr, wo)
    R, S = dev(r), dev(s)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        net.run(R, S, 3, form="gather")
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="relaxed"):
        net.run(R, S, T, form="tensor")
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        for name, ref in (("v", st.v), ("i_syn", st.i_syn), ("v_out", st.v_out), ("counts", st.counts)):
            assert np.array_equal(bits(net.read(name)), bits(ref)), name
    net.close()


@pytest.mark.parametrize("B,NI,N,T,reduce", [
    (3, 7, 1, 60, "mean"),         # one column, fewer inputs than a list's load
    (37, 100, 6007, 8, "sum"),     # 16 columns a block, rows that are not 16-byte aligned, a short last tile
    (65, 30, 2504, 12, "max"),     # eight columns a block, three mask words
    (257, 9, 130, 25, "mean"),     # four columns a block, nine mask words, a last tile of two
])
def test_column_tile_step(B, NI, N, T, reduce):
    """The column-tile step at the edges of its tiles, learning and frozen, and
    handing over to the persistent form and to the separate (profiled) kernels
    in continuing runs."""
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.fig1_workload(B, N, n_in=NI)
    p.update(theta_plus=0.05, w_ei=22.5, w_ie=-0.5, e_thresh=-64.0)     # some inhibition and adaptation
    tp.parity_all_modes(p, r, s, w, T, learn=False, modes=("graph",))
    st, rec = tp.oracle_run(p, r, s, w, T, reduce=reduce)
    assert rec.raster_e.sum() > 0 and np.abs(st.w - w).max() > 0
    net, g = tp.gpu_run(p, r, s, w, T, reduce=reduce, mode="graph")
    tp.assert_parity(g, st, rec)
    for mode in ("step", "persistent", "graph"):
        st, rec = tp.oracle_run(p, r, s, w, 3, reduce=reduce, st=st, episodic=False)
        net, g = tp.gpu_run(p, r, s, w, 3, reduce=reduce, mode=mode, net=net, continue_=True)
        tp.assert_parity(g, st, rec)
    st, rec = tp.oracle_run(p, r, s, w, 2, reduce=reduce, st=st, episodic=False)
    net.run(dev(r), dev(s), 2, reduce=reduce, mode="graph", continue_=True, profile=True)
    assert np.array_equal(net.weights(), st.w) and np.array_equal(net.read("v_exc"), st.v_e)
    net.close()


@pytest.mark.parametrize("B,NI,N,T", [
    (3, 70, 31, 40),         # fewer neurons than a warp, warps without neurons
    (200, 1100, 512, 25),    # the widest layer at one neuron per thread, 35 input words
    (5, 784, 2049, 40),      # four neurons per thread, one of them past a boundary
    (2, 784, 8192, 20),      # the widest layer at eight
])
@pytest.mark.parametrize("wprec", [0, 1, 2])
def test_learning_off_sample_per_cta(B, NI, N, T, wprec):
    """The persistent mode with learning off, after a learning run has left
    traces, so that inputs that never spike decay too; a second continuing run
    has other rates, some of them all zero."""
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.workload(B, N, NI)
    net, g = tp.gpu_run(p, r, s, w, 5, mode="graph", wprec=wprec)
    st, rec = tp.oracle_run(p, r, s, w, 5, wprec=wprec)
    tp.assert_parity(g, st, rec)
    r2 = np.roll(r, 7, axis=1) * np.float32(2)
    r2[0] = 0
    for rates, steps in ((r, T), (r2, 13)):
        st, rec = tp.oracle_run(p, rates, s, w, steps, learn=False, st=st, episodic=False, wprec=wprec)
        net, g = tp.gpu_run(p, rates, s, w, steps, learn=False, mode="persistent", net=net, continue_=True)
        tp.assert_parity(g, st, rec)
    st, rec = tp.oracle_run(p, r, s, w, 4, st=st, episodic=False, wprec=wprec)
    net, g = tp.gpu_run(p, r, s, w, 4, mode="graph", net=net, continue_=True)
    tp.assert_parity(g, st, rec)
    net.close()


@pytest.mark.parametrize("B,NI,N,T,reduce,wprec", [
    (1, 784, 100, 120, "max", 0),      # every sample an event; CTAs of 13 columns, the last short
    (1, 40, 5, 150, "mean", 0),        # fewer columns than CTAs
    (5, 1100, 500, 60, "sum", 1),      # 35 input words, 32 columns a CTA
    (4, 300, 1700, 40, "mean", 0),     # 107 columns: four column rounds, two items a thread
    (11, 300, 620, 60, "mean", 0),     # 39 columns: two column rounds
    (32, 100, 200, 60, "max", 0),      # full masks
])
def test_small_batch_cluster(B, NI, N, T, reduce, wprec):
    """The small-batch learning form, and what it leaves: a continuing run with
    other rates (traces of inputs that no longer spike), then the graph form."""
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.workload(B, N, NI)
    r = np.minimum(r * np.float32(4 * 784 / NI), np.float32(900))       # the oracle fires in every case
    r2 = np.roll(r, 5, axis=1)
    net, st = None, None
    for k, (rates, steps, mode) in enumerate([(r, T, "persistent"), (r2, 30, "persistent"), (r, 10, "graph")]):
        st, rec = tp.oracle_run(p, rates, s, w, steps, reduce=reduce, st=st, episodic=k == 0, wprec=wprec)
        net, g = tp.gpu_run(p, rates, s, w, steps, reduce=reduce, mode=mode, net=net, continue_=k > 0, wprec=wprec)
        tp.assert_parity(g, st, rec)
        assert k > 0 or rec.raster_e.sum() > 0
    net.close()


@pytest.mark.parametrize("B,NI,N,NO", [
    (3, 33, 31, 10),           # 31 bits of the last input word past the inputs
    (2, 1, 700, 3),            # one input; clusters
    (1, 1025, 64, 40),         # 33 input words, more outputs than lanes
])
def test_rec_gather_runs_of_one_step(B, NI, N, NO):
    """Runs of a single step: the closing list, for the readout of that step, holds
    its hidden spikes alone (no input words are drawn for a step after it)."""
    p, r, s, wf, wr, wo = workload(B, NI, N, NO, seed=NI, ff_gain=64.0)
    r = np.full_like(r, 600.0)
    net, st, fired = snn().RecNetwork(p, wf, wr, wo), None, 0
    for t in range(12):
        st, rh, ri = oracle_run(p, r, s, wf, wr, wo, 1, st=st, episodic=t == 0)
        net.run(dev(r), dev(s), 1, continue_=t > 0, record=True, record_input=True, form="gather")
        assert_same(net, st, rh, ri)
        fired += int(rh.sum())
    assert fired > 0
    net.close()


FRESH = """
import sys
sys.path[:0] = [%r, %r]
import numpy as np
import test_gpu_parity as tp
import test_gpu_serving as ts

def workload(B, N, NI):
    p, r, s, w = tp.synth.workload(B, N, NI)
    return p, np.minimum(r * np.float32(4 * 784 / NI), np.float32(900)), s, w
%s
"""
SERVE_ONE = """
p, r, s, w = workload(3, 20, 6032)
m = tp.snn()
net = m.Network(p, w_init=w)
srv = m.snn_serve_create(net.handle, 4, 1 << 30)
ids = {m.snn_serve_submit(srv, r[q], int(s[q]), 30): q for q in range(3)}
while m.snn_serve_status(srv)["active"] or m.snn_serve_status(srv)["queued"]:
    m.snn_serve_step(srv, 11)
m.snn_serve_wait(srv)
for i, c in zip(*m.snn_serve_poll(srv, 20)):
    assert np.array_equal(c, ts.alone_counts(p, w, 0, r[ids[int(i)]], int(s[ids.pop(int(i))]), 30))
assert not ids
"""


@pytest.mark.parametrize("code", [
    "for B in (104, 105, 107, 108): tp.parity_all_modes(*workload(B, 12, 2900), 4, modes=('graph',))",
    "tp.parity_all_modes(*workload(1, 12, 3063), 4, learn=False, modes=('graph',))",
    "for NI in (3997, 3998, 4007, 4008): tp.parity_all_modes(*workload(2, 20, NI), 6, learn=False, modes=('persistent',))",
    SERVE_ONE,
], ids=["column tiles", "column tiles, frozen", "sample per CTA", "serving"])
def test_dynamic_shared_memory_near_the_default_limit(code):
    """The default limit of 48 KB counts a kernel's static shared memory too. In a
    fresh process each: a larger run of the same kernel raises the limit for good."""
    import os
    import subprocess
    import sys
    here = os.path.dirname(os.path.abspath(__file__))
    q = subprocess.run([sys.executable, "-c", FRESH % (os.path.dirname(here), here, code)], capture_output=True, text=True)
    assert q.returncode == 0, q.stderr[-2000:]


@pytest.mark.parametrize("B,NI,N,T,reduce", [
    (3, 120, 1824, 12, "mean"),    # four columns a block: the widest layer whose blocks fit one wave
    (3, 120, 1828, 12, "mean"),    # eight columns: four would need a second wave
    (5, 120, 2031, 12, "sum"),     # the same with unaligned rows and a short last tile
    (514, 100, 1900, 3, "max"),    # four again: the maximum above 512 samples
])
def test_column_tile_step_between_its_tiles(B, NI, N, T, reduce):
    test_column_tile_step(B, NI, N, T, reduce)


def test_column_tile_step_mean_of_columns_without_a_trace():
    """A batch that is no power of two, few columns firing: the mean of the other
    columns' zero sums, and weights at both bounds, for both masters."""
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.workload(7, 203, 120)
    r = np.minimum(r * np.float32(20), np.float32(900))
    w = np.where(np.arange(203) % 5 == 0, w, np.float32(0)).astype(np.float32)
    w[:, 2::10] = 1.0
    for wmaster in (0, 1):
        p.update(wmaster=wmaster)
        st, rec = tp.parity_all_modes(p, r, s, w, 60, modes=("graph", "step"))
        assert rec.raster_e.sum() > 0 and (np.abs(st.w - w).max(0) == 0).any()


@pytest.mark.parametrize("B,NI,N,T,reduce", [
    (1, 97, 5, 40, "max"),         # the fewest inputs, fewer columns than a quad pair
    (257, 100, 130, 12, "mean"),   # four columns a block, nine mask words, a last tile of two
    (65, 120, 2504, 6, "max"),     # eight columns a block, three mask words
    (130, 100, 3653, 4, "sum"),    # several waves, unaligned rows, a short last tile
])
def test_column_tile_step_from_97_inputs(B, NI, N, T, reduce):
    test_column_tile_step(B, NI, N, T, reduce)


@pytest.mark.parametrize("B,NI,N", [
    (128, 100, 40), (129, 100, 40), (100, 100, 1001), (101, 100, 1001), (48, 97, 2441), (49, 97, 2441)])
def test_frozen_steps_on_both_sides_of_the_tiles_line(B, NI, N):
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.fig1_workload(B, N, n_in=NI)
    st, rec = tp.parity_all_modes(p, r, s, w, 40, learn=False, modes=("graph", "step"))
    assert rec.raster_e.sum() > 0


@pytest.mark.parametrize("B,NI,N", [(4096, 100, 50), (2048, 225, 50)])
def test_frozen_steps_of_many_samples_spread_over_the_gpu(B, NI, N):
    """A few blocks that own the columns of all samples took four to eight times as
    long as the separate kernels, which a profiled run launches."""
    m = snn()
    from paper_1909_02549_gb300 import synth
    p, r, s, w = synth.fig1_workload(B, N, n_in=NI)
    net = m.Network(p, w_init=w)
    R, S = dev(r), dev(s)
    best = {}
    for profile in (False, True):
        ms = []
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            net.run(R, S, 50, learn=False, mode="graph", profile=profile)
            e1.record()
            torch.cuda.synchronize()
            ms.append(e0.elapsed_time(e1))
        best[profile] = min(ms)
    net.close()
    assert best[False] < 1.5 * best[True], best


@pytest.mark.parametrize("B,NI,N,wprec", [
    (64, 60, 8192, 0), (64, 60, 8192, 1),      # the widest layer at eight neurons per thread
    (65, 130, 5003, 0), (65, 130, 5003, 1),    # a ragged one
    (70, 60, 4097, 2),                         # FP8: the column kernel
    (153, 40, 4200, 0),                        # one sample past a wave: the column kernel
    (247, 40, 4200, 1),                        # a second wave five eighths full
])
def test_learning_off_wide_layers(B, NI, N, wprec):
    """Eight neurons per thread (64 samples and more) and its limits: a learning run, a
    frozen run that continues it with traces to decay, and another learning one."""
    import test_gpu_parity as tp
    import oracle
    import os
    oracle.set_threads(os.cpu_count() or 1)
    p, r, s, w = tp.synth.workload(B, N, NI)
    r = np.minimum(r * np.float32(4 * 784 / NI), np.float32(900))
    r2 = np.roll(r, 7, axis=1)
    r2[0] = 0
    net, st = None, None
    for k, (rates, steps, learn, mode) in enumerate([(r, 3, True, "graph"), (r2, 25, False, "persistent"), (r, 2, True, "graph")]):
        st, rec = tp.oracle_run(p, rates, s, w, steps, learn=learn, st=st, episodic=k == 0, wprec=wprec)
        net, g = tp.gpu_run(p, rates, s, w, steps, learn=learn, mode=mode, net=net, continue_=k > 0, wprec=wprec)
        tp.assert_parity(g, st, rec)
        assert k != 1 or rec.raster_e.sum() > 0
    net.close()
    oracle.set_threads(1)


@pytest.mark.parametrize("B,NI,N,reduce", [
    (32, 100, 144, "mean"), (32, 100, 145, "mean"),    # 288 items a CTA, and more: the column kernel
    (24, 60, 112, "mean"), (24, 60, 113, "mean"),      # divided means: 168
    (14, 40, 256, "max"), (1, 40, 4608, "sum"), (1, 40, 4609, "sum"),
])
def test_small_batch_without_inhibition(B, NI, N, reduce):
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.fig1_workload(B, N, n_in=NI)
    r = r * np.float32(100 / NI)
    st, rec = tp.parity_all_modes(p, r, s, w, 60, reduce=reduce, modes=("persistent",))
    assert rec.raster_e.sum() > 0 and np.abs(st.w - w).max() > 0


@pytest.mark.parametrize("wprec", [0, 1, 2])
def test_narrow_column_kernel_rows_past_the_staged_ones(wprec):
    """One column a CTA, samples with hundreds of active inputs (odd and even counts):
    most of a sample's rows come from the list's part that is not staged."""
    import test_gpu_parity as tp
    B, NI, N = 600, 1023, 130
    p, r, s, w = tp.synth.workload(B, N, NI)
    r = np.minimum(r * np.float32(12), np.float32(900))
    st, rec = tp.parity_all_modes(p, r, s, w, 6, reduce="sum", modes=("persistent",), wprec=wprec)
    assert rec.raster_e.sum() > 0 and (r > 0).sum(1).max() > 300


@pytest.mark.parametrize("B,NI,N", [(1, 64, 2048), (2, 33, 4000), (9, 30, 7700)])
def test_rec_tensor_form_of_a_few_samples_in_coarser_parts(B, NI, N):
    """Wide layers whose operand is small: halves instead of quarters, whole tiles
    instead of halves."""
    test_rec_tensor_form_cut_tiles(B, NI, N, 10)


@pytest.mark.parametrize("T,folds", [(1, 1), (31, 1), (32, 2), (62, 2), (63, 3)])
def test_rec_profile_brackets_the_spike_counts(T, folds):
    p, r, s, wf, wr, wo = dyadic_workload(4, 64, 96, 10, seed=23)
    net = snn().RecNetwork(p, wf, wr, wo)
    for form, n in (("tensor", folds), ("gather", 0)):
        net.run(dev(r), dev(s), T, form=form, profile=True)
        prof = net.profile()
        assert prof["counts"][1] == n and (prof["counts"][0] > 0) == (n > 0), prof
        assert prof["drive"][1] == T
    net.close()


@pytest.mark.parametrize("N,wprec", [(1000, 0), (1000, 2), (3000, 0), (3000, 1), (5000, 0), (8200, 0), (8200, 1)])
def test_serving_wider_layers(N, wprec):
    """Two, four and eight neurons per thread, and the kernel of the layers too wide
    for registers: requests of several calls with retirements inside them."""
    import test_gpu_serving as ts
    from paper_1909_02549_gb300 import synth
    m, NI, nreq = snn(), 100, 7
    p, r, s, w = synth.workload(nreq, N, NI)
    r = np.minimum(r * np.float32(30), np.float32(900))
    net = m.Network(p, w_init=w, wprec=wprec)
    srv = m.snn_serve_create(net.handle, 3, 1 << 30)
    ids = {m.snn_serve_submit(srv, r[q], int(s[q]), 21 + 5 * q): q for q in range(nreq)}
    while m.snn_serve_status(srv)["active"] or m.snn_serve_status(srv)["queued"]:
        m.snn_serve_step(srv, 8)
    m.snn_serve_wait(srv)
    done, counts = m.snn_serve_poll(srv, N, max_n=nreq)
    m.snn_serve_destroy(srv)
    assert sorted(int(i) for i in done) == sorted(ids) and counts.sum() > 0
    for i, c in zip(done, counts):
        q = ids[int(i)]
        assert np.array_equal(c, ts.alone_counts(p, w, wprec, r[q], int(s[q]), 21 + 5 * q)), q
    net.close()


@pytest.mark.parametrize("B,NI,N", [(1, 120, 60), (5, 784, 300)])
def test_small_batch_runs_of_a_few_steps(B, NI, N):
    """Continuing runs of one to nine steps, the column kernel's and the cluster's."""
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.workload(B, N, NI)
    r = np.minimum(r * np.float32(4 * 784 / NI), np.float32(900))
    net, st, fired = None, None, 0
    for k, T in enumerate((1, 2, 3, 4, 5, 6, 7, 8, 9, 30, 1)):
        st, rec = tp.oracle_run(p, r, s, w, T, st=st, episodic=k == 0)
        net, g = tp.gpu_run(p, r, s, w, T, mode="persistent", net=net, continue_=k > 0)
        tp.assert_parity(g, st, rec)
        fired += int(rec.raster_e.sum())
    assert fired > 0
    net.close()


@pytest.mark.parametrize("B,NI,N", [(64, 100, 1028), (128, 100, 1028)])
def test_column_tile_step_runs_of_one_step(B, NI, N):
    import test_gpu_parity as tp
    p, r, s, w = tp.synth.fig1_workload(B, N, n_in=NI)
    net, st = None, None
    for k, T in enumerate((40, 1, 1, 2, 1)):
        st, rec = tp.oracle_run(p, r, s, w, T, st=st, episodic=k == 0)
        net, g = tp.gpu_run(p, r, s, w, T, mode=("graph", "step")[k & 1], net=net, continue_=k > 0)
        tp.assert_parity(g, st, rec)
        assert k > 0 or rec.raster_e.sum() > 0
    net.close()
