"""GPU parity of the dense resident engine (small networks of dense edges and small convolutions: weights and states in the shared
memory of one thread-block cluster, all frames of a run in one launch) against the oracle, and its hand-over to the per-frame
launch path: states left in global memory, frame counter, resumed runs."""
import numpy as np
import pytest

from tests import parity
from workloads import data, graphs
from workloads.graphs import CONV, DENSE, GAP_DENSE, IDENTITY, RELU, Edge, GraphSpec, Node, sequential_pattern, streaming_pattern

pytestmark = pytest.mark.gpu

# CTAs per cluster: sixteen when a frame is one tableau level (streaming), eight otherwise
CLUSTER = {"streaming": 16, "sequential": 8, "hybrid": 8}


def mlp(batch, frames, sizes=(36, 20, 10, 7), seed=31):
    """input -> h1 -> h2 -> out with a skip input -> out, a self-loop on h2 and a back-edge h2 -> h1."""
    nodes = [Node("in", 1, 1, sizes[0], IDENTITY), Node("h1", 1, 1, sizes[1], RELU), Node("h2", 1, 1, sizes[2], RELU),
             Node("out", 1, 1, sizes[3], IDENTITY)]
    edges = [Edge(0, 1, DENSE), Edge(1, 2, DENSE), Edge(2, 3, DENSE), Edge(0, 3, GAP_DENSE), Edge(2, 2, DENSE), Edge(2, 1, DENSE)]
    g = GraphSpec("mlp", nodes, edges, batch=batch, frames=frames, dtype="fp32", seed=seed, weight_gain=1.0)
    g.patterns = {"streaming": streaming_pattern(g), "sequential": sequential_pattern(g), "hybrid": [0, 1, 0, 1, 1, 1]}
    return g


@pytest.mark.parametrize("pattern", ["streaming", "sequential"])
def test_c1_runs_on_the_dense_resident_engine(pattern):
    g = graphs.build("c1")
    cluster = CLUSTER[pattern]
    parity.check_run(g, pattern, expect_resident=cluster)
    parity.check_run(g, pattern, frames=1, expect_resident=cluster)
    parity.check_run(g, pattern, resident=False, expect_resident=0)


@pytest.mark.parametrize("batch", [1, 8, 11, 40])
def test_odd_sizes_and_batches(batch):
    # channel counts that are no multiple of four (padded columns), more sequences than one cluster holds, a ragged last cluster
    g = mlp(batch, 7)
    for p in g.patterns:
        parity.check_run(g, p, expect_resident=CLUSTER[p])


def test_runs_and_steps_continue_each_other():
    import torch
    from oracle import frame_update as fu
    g = mlp(5, 12)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "streaming", X, W, Bi)
    G = parity.make_graph(g, "streaming", "auto", 0, W, Bi)
    assert G.info["resident_cluster"] == CLUSTER["streaming"]
    x = parity.to_device(g, X[0])
    G.reset([x[0]])
    out = torch.empty((4, 5, 7), dtype=torch.float32, device="cuda:0")
    G.run([x[1:5]], out)                              # resident: frames 1..4
    assert G.frame() == 4
    for t in (5, 6):                                   # launch path continues from the states the kernel left
        G.step([x[t]])
    G.run([x[7:11]], out)                              # resident again: frames 7..10
    G.step([x[11]])
    G.run([x[12:13]], out[:1])
    G.sync_status()
    assert G.frame() == 12
    o = G.output_node
    assert parity.rel_err(out[:1].cpu().numpy().reshape(want[o][12:13].shape), want[o][12:13]) <= 1e-4
    for v in range(len(g.nodes)):
        assert parity.rel_err(G.get_state(v).cpu().numpy(), want[v][12]) <= 1e-4, g.nodes[v].name


def test_results_are_reproducible_bit_for_bit():
    g = graphs.build("c1")
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g)
    outs = []
    for _ in range(2):
        G = parity.make_graph(g, "streaming", "auto", 0, W, Bi)
        outs.append(G.rollout([parity.to_device(g, X[0])]).cpu().numpy())
    assert np.array_equal(outs[0], outs[1])


@pytest.mark.parametrize("batch", [1, 3, 15, 28, 130])
def test_sequences_per_cluster_and_ranks_without_rows(batch):
    # few rows: most CTAs of a cluster have no work unit in a level and only take part in the exchange; the batches make clusters
    # of two, four and eight sequences (and, the last, more clusters of sixteen CTAs than a device holds), the last one ragged
    g = mlp(batch, 6, sizes=(4, 3, 2, 5), seed=77)
    for p in g.patterns:
        parity.check_run(g, p, expect_resident=8 if batch == 130 else CLUSTER[p])


@pytest.mark.parametrize("batch", [1, 9, 260])
def test_single_steps(batch):
    # frame by frame: on the engine, but for a frame that starts off a 16-byte boundary and for a batch of several waves (260)
    import torch
    from oracle import frame_update as fu
    g = mlp(batch, 5)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    for p in ("streaming", "sequential"):
        want = fu.rollout_spec(g, p, X, W, Bi)
        G = parity.make_graph(g, p, "auto", 0, W, Bi)
        x = parity.to_device(g, X[0])
        odd = torch.empty(x[3].numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x[3].shape).copy_(x[3])
        assert odd.data_ptr() % 16 != 0
        G.reset([x[0]])
        out = torch.empty((5,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
        for t in range(1, 6):
            G.step([odd if t == 3 else x[t]], out[t - 1])
        G.sync_status()
        o = G.output_node
        assert parity.rel_err(out.cpu().numpy().reshape(want[o][1:6].shape), want[o][1:6]) <= 1e-4
        for v in range(len(g.nodes)):
            assert parity.rel_err(G.get_state(v).cpu().numpy(), want[v][5]) <= 1e-4, g.nodes[v].name


@pytest.mark.parametrize("pattern", ["streaming", "sequential"])
@pytest.mark.parametrize("batch", [8, 64, 128])
def test_a_smaller_network_leaves_a_larger_one_runnable(pattern, batch):
    # both run on the same kernels (cluster size and sequences per cluster follow from batch and pattern), whose shared-memory limit
    # they share; the larger network runs before and after the smaller one was planned and run
    import torch
    from oracle import frame_update as fu
    g, small = graphs.build("c1", batch=batch, frames=4), mlp(batch, 4)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    samples = [0, batch - 1]
    want = fu.rollout_spec(g, pattern, X, W, Bi, samples=samples)
    G = parity.make_graph(g, pattern, "auto", 0, W, Bi)
    x, o = parity.to_device(g, X[0]), G.output_node
    for _ in range(2):
        out = torch.empty((4,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
        G.reset([x[0]])
        G.run([x[1:3]], out[:2])
        for t in (3, 4):
            G.step([x[t]], out[t - 1])
        G.sync_status()
        assert parity.rel_err(out.cpu().numpy()[:, samples].reshape(want[o][1:].shape), want[o][1:]) <= 1e-4
        parity.check_run(small, pattern, samples=samples)
        parity.check_stepwise(small, pattern, samples=samples)


def small_cnn(batch, frames, dtype, cin=1, size=(12, 10), c=12, seed=41):
    """input -> a (5x5, stride 2, recurrent) -> b (3x3), both -> h (dense) -> out, skips a -> out, input -> b (1x1, stride 2)."""
    h, w = size
    nodes = [Node("in", h, w, cin, IDENTITY), Node("a", h // 2, w // 2, c, RELU), Node("b", h // 2, w // 2, 8, RELU), Node("h", 1, 1, 22, RELU),
             Node("out", 1, 1, 7, IDENTITY)]
    edges = [Edge(0, 1, CONV, 5, 2), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(0, 2, CONV, 1, 2), Edge(1, 3, DENSE), Edge(2, 3, DENSE),
             Edge(3, 4, DENSE), Edge(1, 4, DENSE), Edge(3, 3, DENSE)]
    g = GraphSpec("small_cnn", nodes, edges, batch=batch, frames=frames, dtype=dtype, seed=seed, weight_gain=1.0)
    g.patterns = {"streaming": streaming_pattern(g), "sequential": sequential_pattern(g), "hybrid": [0, 1, 1, 0, 0, 1, 0, 1, 1]}
    return g


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,cin,size,c", [(1, 1, (12, 10), 12), (3, 3, (12, 8), 4), (8, 4, (6, 10), 32), (11, 1, (14, 14), 16), (41, 2, (8, 8), 20)])
def test_small_convolutions(dtype, batch, cin, size, c):
    # blocks of eight quads that are not full, sources of one to many channels, ragged clusters; sixteen-bit states are rounded as the
    # launch path rounds them
    g = small_cnn(batch, 6, dtype, cin, size, c)
    for p in g.patterns:
        parity.check_run(g, p)
        parity.check_run(g, p, frames=1)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_small_networks_run_on_the_engine_in_both_types(dtype):
    g = mlp(5, 4)
    g.dtype = dtype
    for p in g.patterns:
        parity.check_run(g, p, expect_resident=CLUSTER[p])
        parity.check_stepwise(g, p, zero_bias=False)
    g = small_cnn(5, 5, dtype)
    for p in g.patterns:
        parity.check_run(g, p, expect_resident=CLUSTER[p])
        parity.check_stepwise(g, p, zero_bias=False)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_convolutions_hand_over_to_the_launch_path_and_back(dtype):
    import torch
    from oracle import frame_update as fu
    g = small_cnn(5, 12, dtype)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "sequential", X, W, Bi)
    G = parity.make_graph(g, "sequential", "auto", 0, W, Bi)
    x = parity.to_device(g, X[0])
    shifted = torch.empty(x[5:7].numel() + 1, dtype=x.dtype, device="cuda:0")[1:].view(x[5:7].shape)   # not on a 16-byte boundary:
    shifted.copy_(x[5:7])                                                                               # the launch path takes it
    out = torch.empty((11, 5, 7), dtype=torch.float32, device="cuda:0")
    G.reset([x[0]])
    G.run([x[1:5]], out[:4])
    G.run([shifted], out[4:6])
    G.run([x[7:12]], out[6:])
    G.sync_status()
    assert parity.rel_err(out.cpu().numpy(), want[4][1:12].reshape(11, 5, 7)) <= parity.TOL[dtype]
    for v in range(5):
        assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][11]) <= parity.TOL[dtype]


@pytest.mark.parametrize("pattern", ["streaming", "sequential"])
@pytest.mark.parametrize("batch,width", [(72, 784), (67, 1000), (9, 4)])
def test_bf16_input_frames_of_more_vectors_than_the_fetching_threads_hold(pattern, batch, width):
    # with eight sequences per cluster a frame of the 784-wide input is up to 17 vectors for each of 96 fetching threads, which have
    # eight on their way at a time; the last cluster is not full
    g = mlp(batch, 5, (width, 128, 128, 10))
    g.dtype = "bf16"
    samples = sorted({0, 7, batch // 2, batch - 1})
    parity.check_run(g, pattern, samples=samples, expect_resident=CLUSTER[pattern] if batch == 9 else 8)
    parity.check_run(g, pattern, samples=samples, frames=2)


@pytest.mark.parametrize("dtype,pattern,batch,resident", [
    ("fp32", "streaming", 32, True), ("fp32", "streaming", 400, False), ("fp32", "sequential", 32, True), ("fp32", "sequential", 800, False),
    ("bf16", "streaming", 2, True), ("bf16", "streaming", 400, False), ("bf16", "sequential", 400, False),
])
def test_convolutions_in_more_waves_than_pay_are_launched(dtype, pattern, batch, resident):
    # one wave of clusters, in fp32 two where a frame is several launches; a device holds 18 clusters of eight CTAs at most
    g = small_cnn(batch, 3, dtype)
    G = parity.make_graph(g, pattern, "auto", 0, data.make_weights(g), data.make_biases(g))
    assert (G.info["resident_cluster"] > 0) == resident, G.info
    samples = sorted({0, batch // 2, batch - 1})
    parity.check_run(g, pattern, samples=samples)


def test_staged_copies_are_brought_up_to_date_behind_the_engine():
    # a few-channel input edge that the launch path reads through staged copies of the frame before, which neither a reset nor the engine
    # writes: frames from a buffer that is not on a 16-byte boundary, which the engine does not take, follow each of them
    import torch
    from oracle import frame_update as fu
    g = small_cnn(5, 14, "bf16", 3, (12, 12), 16)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "streaming", X, W, Bi)
    G = parity.make_graph(g, "streaming", "auto", 0, W, Bi)
    assert G.info["resident_cluster"] == CLUSTER["streaming"] and G.info["n_tensor_core_nodes"] == 1
    x = parity.to_device(g, X[0])

    def shifted(a):
        y = torch.empty(a.numel() + 1, dtype=a.dtype, device="cuda:0")[1:].view(a.shape)
        return y.copy_(a)

    def check(t):
        G.sync_status()
        for v in range(5):
            assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][t]) <= parity.TOL["bf16"], (v, t)

    G.reset([x[0]])
    G.run([shifted(x[1:3])])             # a reset, then launches
    check(2)
    G.run([x[3:6]])
    G.run([shifted(x[6:8])])             # a run of the engine, then launches
    check(7)
    G.step([x[8]])
    G.step([shifted(x[9])])              # a step of the engine, then a launched one
    check(9)
    G.step([x[10]])
    G.run([shifted(x[11:13])])
    check(12)
    G.reset([x[0]])
    G.step([shifted(x[1])])
    check(1)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,cin,size,c", [(1, 1, (12, 10), 12), (3, 3, (12, 8), 4), (8, 4, (6, 10), 32), (11, 1, (14, 14), 16), (41, 2, (8, 8), 20)])
def test_small_convolutions_take_the_engine(dtype, batch, cin, size, c):
    # (in bf16 with more than four sequences per cluster, which 41 take, frames of one level are launched)
    g = small_cnn(batch, 6, dtype, cin, size, c)
    for p in g.patterns:
        on_chip = 0 if dtype == "bf16" and p == "streaming" and batch == 41 else CLUSTER[p]
        G = parity.make_graph(g, p, "auto", 0, data.make_weights(g), data.make_biases(g))
        assert G.info["resident_cluster"] == on_chip, (p, G.info)
