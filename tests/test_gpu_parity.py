"""GPU parity: the CUDA library, called through the C ABI, against the CPU oracle on the same
seeded inputs.  Tolerances: max-abs-diff relative to each node's output scale, 2e-2 for bfloat16
states, 1e-4 for fp32; the dyadic worked example must match exactly."""
import numpy as np
import pytest

from tests import parity
from workloads import data, graphs

pytestmark = pytest.mark.gpu


def test_worked_example_exact():
    import torch
    from paper_1806_04965_b200 import Graph
    g = graphs.worked_example()
    x = torch.tensor([1, 2, 0, 3, 1], dtype=torch.float32, device="cuda:0").reshape(5, 1, 1, 1, 1)
    w = [np.array(v, dtype=np.float32).reshape(1, 1, 1, 1) for v in (1, 0.5, 2, -1)]
    b = [np.zeros(1, np.float32), np.array([-0.5], np.float32), np.array([0.25], np.float32)]
    want = {"streaming": [(0.5, 0), (1.75, 0), (0.375, 3.75), (2.6875, 0)],
            "sequential": [(1.5, 1.25), (0.25, 0.75), (2.625, 2.5), (1.8125, 2.875)],
            "hybrid": [(1.5, 0), (0.25, 3.25), (2.625, 0), (1.8125, 4.5)]}
    for dtype in ("fp32", "bf16"):
        for p, R in g.patterns.items():
            G = Graph(g.nodes, g.edges, R, batch=1, dtype=dtype)
            G.set_weights(w, b)
            xs = x if dtype == "fp32" else x.to(torch.bfloat16)
            G.reset([xs[0]])
            got = []
            for t in range(1, 5):
                G.step([xs[t]])
                got.append((float(G.get_state(1).float().item()), float(G.get_state(2).float().item())))
            assert got == [(float(a), float(c)) for (a, c) in want[p]], (dtype, p, got)


@pytest.mark.parametrize("pattern", ["streaming", "sequential"])
def test_c1_mlp_full_size(pattern):
    parity.check_stepwise(graphs.build("c1"), pattern)
    parity.check_run(graphs.build("c1"), pattern)
    parity.check_run(graphs.build("c1"), pattern, graph_frames=4)


@pytest.mark.parametrize("kind", ["FF", "S", "SR"])
def test_paper_mnist_networks_fp32(kind):
    g = graphs.mnist_net(kind, batch=3, frames=5)
    for p in g.patterns:
        parity.check_stepwise(g, p, zero_bias=False)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("name,kw", [
    ("c2", dict(batch=3, frames=6)),
    ("c3", dict(batch=2, frames=4, size=16)),
    ("c4", dict(batch=2, frames=4, size=16)),
    ("c5", dict(batch=2, frames=4, size=16)),
])
def test_configs_reduced_direct_engine(name, kw, dtype):
    g = graphs.build(name, dtype=dtype, **kw)
    for p in g.patterns:
        parity.check_stepwise(g, p, engine="direct", zero_bias=False)


def test_run_equals_steps_and_resume():
    import torch
    g = graphs.build("c2", batch=4, frames=8, dtype="fp32")
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    A = parity.make_graph(g, "streaming", "direct", 0, W, Bi)
    Bg = parity.make_graph(g, "streaming", "direct", 3, W, Bi)
    x = parity.to_device(g, X[0])
    oa = A.rollout([x])
    ob = Bg.rollout([x])                     # CUDA graphs of 3 frames + 2 plain frames
    assert torch.equal(oa, ob)
    # resume: run 4 frames, move every state into a fresh graph, run the other 4
    C = parity.make_graph(g, "streaming", "direct", 0, W, Bi)
    C.reset([x[0]])
    C.run([x[1:5]])
    D = parity.make_graph(g, "streaming", "direct", 0, W, Bi)
    D.reset([x[4]])
    for v in range(len(g.nodes)):
        D.set_state(v, C.get_state(v))
    od = torch.empty((4, g.batch, 10), dtype=torch.float32, device="cuda:0")
    D.run([x[5:9]], od)
    assert torch.equal(od, oa[4:])
    assert A.launch_count() > 0


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_spatial_output_node_fills_a_full_frame(dtype):
    # the output node is an image: `out` holds [B][H][W][C] floats per frame, and consecutive frames of a run do not overlap
    import torch
    g = graphs.build("sink", dtype=dtype)
    for p in g.patterns:
        parity.check_stepwise(g, p, zero_bias=False)
        parity.check_run(g, p)
    from paper_1806_04965_b200 import Graph
    G = Graph(g.nodes, g.edges, g.patterns["streaming"], batch=g.batch, dtype=dtype)
    assert G.out_shape() == (g.batch, 4, 4, 8)
    G.set_weights(data.make_weights(g), data.make_biases(g, zero=False))
    X = data.make_inputs(g)
    # guard words behind the output buffer stay untouched
    buf = torch.full((g.frames * g.batch * 4 * 4 * 8 + 64,), 7.0, dtype=torch.float32, device="cuda:0")
    out = buf[:g.frames * g.batch * 4 * 4 * 8].view(g.frames, g.batch, 4, 4, 8)
    x = parity.to_device(g, X[0])
    G.reset([x[0]])
    G.run([x[1:]], out)
    G.sync_status()
    assert bool((buf[-64:] == 7.0).all())
    assert float(out.abs().max()) > 0


def test_expired_device_wait_is_reported_and_cleared_by_reset():
    # host-side hook only: with a wait limit of zero every tensor-core launch reports the expiry at its entry and
    # returns before it touches a barrier, a copy or an MMA; nothing on the GPU actually waits
    from paper_1806_04965_b200 import SrError
    g = graphs.build("c3", batch=2, frames=3, size=16)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g)
    G = parity.make_graph(g, "streaming", "auto", 0, W, Bi, wait_limit_ms=0)
    assert G.info["n_tensor_core_nodes"] > 0 and G.info["resident_cluster"] == 0
    x = parity.to_device(g, X[0])
    G.rollout([x])
    for _ in range(2):                                  # the error stays recorded until the rollout starts over
        with pytest.raises(SrError) as e:
            G.sync_status()
        assert e.value.status == "SR_ERR_TIMEOUT"
    G.set_option(10, 1000)
    want = fu_rollout(g, X, W, Bi)
    out = G.rollout([x])                                # reset clears the error word
    G.sync_status()
    o = G.output_node
    assert parity.rel_err(out.cpu().numpy().reshape(want[o][1:].shape), want[o][1:]) <= parity.TOL["bf16"]
    parity.check_run(g, "streaming")                    # and a fresh graph is unaffected


def fu_rollout(g, X, W, Bi):
    from oracle import frame_update as fu
    return fu.rollout_spec(g, "streaming", X, W, Bi)


@pytest.mark.parametrize("name,kw,W", [("c4ff", dict(batch=3, frames=9, size=16), 4), ("dsr2", dict(batch=2, frames=7, h1_recurrence=False), 3),
                                        ("mini_ff", dict(), 5)])
def test_deep_window_equals_chained_windows(name, kw, W):
    # a network without recurrence under the sequential rollout: the W frames of a window do not depend on each other and
    # are evaluated at once (one launch group per level over W * B samples); results equal W single steps, the graph
    # stands at frame t + W afterwards and can be stepped on (two windows, then single steps to the end)
    import torch
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, sequential_pattern, streaming_pattern
    if name == "mini_ff":
        # a streaming input edge (reads the previous input frame) beside within-frame edges
        nodes = [Node("in", 16, 16, 3, IDENTITY), Node("a", 16, 16, 32), Node("b", 8, 8, 64), Node("o", 1, 1, 5, IDENTITY)]
        edges = [Edge(0, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 2), Edge(0, 2, CONV, 1, 2), Edge(2, 3, GAP_DENSE)]
        g = GraphSpec("mini_ff", nodes, edges, batch=3, frames=12, dtype="bf16", seed=77)
        g.patterns = {"sequential": [0, 0, 1, 0]}
    elif name == "dsr2":
        g = graphs.dsr(2, **kw)
    else:
        g = graphs.build(name, **kw)
    from oracle import frame_update as fu
    X, Wt, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "sequential", X, Wt, Bi)
    G = parity.make_graph(g, "sequential", "auto", 0, Wt, Bi)
    G.bind_window(W)
    x = {v: parity.to_device(g, X[v]) for v in G.input_nodes}
    G.reset([x[v][0] for v in G.input_nodes])
    o, tol = G.output_node, parity.TOL[g.dtype]
    t = 0
    for _ in range(2):
        out = torch.empty((W,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
        G.rollout_window([x[v][t + 1:t + 1 + W] for v in G.input_nodes], out)
        assert G.frame() == t + W
        assert parity.rel_err(out.cpu().numpy().reshape(want[o][t + 1:t + 1 + W].shape), want[o][t + 1:t + 1 + W]) <= tol
        t += W
        for v in range(len(g.nodes)):
            assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][t]) <= tol, (g.nodes[v].name, t)
    while t < g.frames:
        G.step([x[v][t + 1] for v in G.input_nodes])
        t += 1
        for v in range(len(g.nodes)):
            assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][t]) <= tol, (g.nodes[v].name, t)
    G.sync_status()


def test_deep_window_refuses_patterns_with_recurrence():
    from paper_1806_04965_b200 import SrError
    g = graphs.build("c2", batch=2, frames=3)
    G = parity.make_graph(g, "streaming", "auto", 0, data.make_weights(g), data.make_biases(g))
    with pytest.raises(SrError) as e:
        G.bind_window(4)
    assert e.value.status == "SR_ERR_UNSUPPORTED"


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_edges_that_bridge_several_frames_run_as_chains_of_copy_nodes(dtype):
    # Sec. 6: R(e) > 1 is covered through copy-nodes.  The library takes patterns with values in {0, 1}; the expanded
    # graph (identity 1x1 copies, one frame per link) must reproduce the oracle's direct evaluation of the delays, on the
    # tensor cores (64-channel nodes, bf16) as on the CUDA cores (fp32).
    from oracle import frame_update as fu
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node
    g = GraphSpec("delays", [Node("in", 16, 16, 3, IDENTITY), Node("a", 16, 16, 64), Node("b", 8, 8, 64), Node("o", 1, 1, 5, IDENTITY)],
                  [Edge(0, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 2), Edge(2, 2, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(0, 2, CONV, 1, 2),
                   Edge(2, 3, GAP_DENSE)], batch=3, frames=7, dtype=dtype, seed=77)
    delays = [1, 1, 2, 3, 2, 1]                        # b's recurrence bridges 2 frames, a's 3, the skip from the input 2
    g.patterns["delayed"] = delays
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "delayed", X, W, Bi)
    ex, ident = graphs.with_copy_nodes(g, delays)
    assert len(ex.nodes) == len(g.nodes) + 4
    W_ex = list(W) + [np.eye(c, dtype=np.float32).reshape(c, 1, 1, c) for c in ident]
    B_ex = list(Bi) + [np.zeros(n.c, dtype=np.float32) for n in ex.nodes[len(g.nodes):]]
    G = parity.make_graph(ex, "p", "auto", 0, W_ex, B_ex)
    if dtype == "bf16":
        assert G.info["n_tensor_core_nodes"] >= 2, G.info
    out = G.rollout([parity.to_device(ex, X[0])])
    G.sync_status()
    o = G.output_node
    assert o == 3
    tol = parity.TOL[dtype]
    assert parity.rel_err(out.cpu().numpy().reshape(want[o][1:].shape), want[o][1:]) <= tol
    for v in range(len(g.nodes)):
        assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][g.frames]) <= tol, g.nodes[v].name


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch", [1, 15, 16, 19])
@pytest.mark.parametrize("c_mid,c_out", [(9, 1), (32, 17)])
def test_heads_at_the_edges_of_their_blocks(batch, c_mid, c_out, dtype):
    # dense nodes take 4 samples x 8 outputs per block from 16 samples on, 1 x 2 below; reductions of 4 x 4 x 12 = 192, of 1100
    # (more than one step of 256 threads) and of c_mid (not a multiple of four: scalar loads); a node with a mean-dense
    # edge sums two means and a dense edge.  Tolerance: that of the element type, as everywhere.
    from workloads.graphs import CONV, DENSE, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    nodes = [Node("in", 4, 4, 12, IDENTITY), Node("flat", 1, 1, 1100, IDENTITY), Node("a", 1, 1, c_mid), Node("m", 1, 1, 6), Node("o", 1, 1, c_out, IDENTITY)]
    edges = [Edge(0, 2, DENSE), Edge(1, 2, DENSE), Edge(2, 2, DENSE), Edge(0, 3, GAP_DENSE), Edge(1, 3, DENSE), Edge(0, 3, GAP_DENSE),
             Edge(2, 4, DENSE), Edge(3, 4, DENSE)]
    g = GraphSpec("heads", nodes, edges, batch=batch, frames=3, dtype=dtype, seed=88)
    check_shapes(g)
    g.patterns = {"p": [1] * 8, "q": [0, 1, 1, 0, 0, 1, 0, 0]}
    for p in g.patterns:
        parity.check_stepwise(g, p, zero_bias=False, resident=False)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,classes", [(1, 1), (1, 300), (3, 65), (37, 17), (150, 9), (150, 41)])
def test_mean_heads_in_several_blocks(batch, classes, dtype):
    # blocks of 8, 16, ... outputs with a ragged last one.  m: two means and a dense edge of K % 4 == 0; s: a dense edge of odd K;
    # w1: channels that are no multiple of four, fewer and more than threads; w2: more channels than a block's means, alone and
    # beside others; w3: more than six edges, dense and mean.  R = 0 edges read the frame's own input.
    from workloads.graphs import CONV, DENSE, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    nodes = [Node("in", 4, 4, 12, IDENTITY), Node("odd", 3, 3, 9, IDENTITY), Node("wide", 2, 2, 1028, IDENTITY), Node("m", 1, 1, classes),
             Node("s", 1, 1, 5), Node("w1", 1, 1, classes), Node("w2", 1, 1, classes, IDENTITY), Node("w3", 1, 1, classes), Node("big", 1, 1, 301),
             Node("w4", 1, 1, 6, IDENTITY), Node("o", 1, 1, 3, IDENTITY)]
    edges = [Edge(0, 3, GAP_DENSE), Edge(0, 3, DENSE), Edge(0, 3, GAP_DENSE), Edge(0, 4, GAP_DENSE), Edge(1, 4, DENSE), Edge(1, 5, GAP_DENSE),
             Edge(0, 5, GAP_DENSE), Edge(2, 6, GAP_DENSE), Edge(1, 6, GAP_DENSE)]
    edges += [Edge(i % 2, 7, GAP_DENSE if i % 3 else DENSE) for i in range(9)]
    edges += [Edge(0, 8, DENSE), Edge(8, 9, GAP_DENSE), Edge(2, 9, DENSE)] + [Edge(v, 10, DENSE) for v in (3, 4, 5, 6, 7, 9)]
    g = GraphSpec("heads", nodes, edges, batch=batch, frames=3, dtype=dtype, seed=89)
    check_shapes(g)
    g.patterns = {"p": [1] * len(edges), "q": [i % 2 for i in range(len(edges))]}
    for p in g.patterns:
        parity.check_stepwise(g, p, zero_bias=False, resident=False, samples=[0, batch - 1])
        parity.check_run(g, p, graph_frames=2, resident=False, samples=[0, batch - 1])


def test_states_after_a_deep_window():
    # the states a window leaves behind can be read, replaced one by one, and are superseded by the next update
    import torch
    from oracle import frame_update as fu
    g = graphs.dsr(2, batch=2, frames=5, h1_recurrence=False)
    X, Wt, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "sequential", X, Wt, Bi)
    G = parity.make_graph(g, "sequential", "auto", 0, Wt, Bi)
    G.bind_window(2)
    x = parity.to_device(g, X[0])
    G.reset([x[0]])

    def check(t, skip=-1):
        for v in range(len(g.nodes)):
            if v != skip:
                assert parity.rel_err(G.get_state(v).float().cpu().numpy(), want[v][t]) <= parity.TOL[g.dtype], (t, g.nodes[v].name)

    for t in (0, 2):
        G.rollout_window([x[t + 1:t + 3]])
        check(t + 2)
    mark = torch.full_like(G.get_state(2), 3.0)
    G.set_state(2, mark)
    assert torch.equal(G.get_state(2), mark)
    check(4, skip=2)
    G.step([x[5]])
    check(5)
    G.reset([x[0]])
    assert float(G.get_state(2).abs().max()) == 0.0


def test_expired_wait_in_a_deep_window_is_reported():
    # the host-side hook of a zero wait limit, set once the window is bound: nothing on the GPU actually waits
    import torch
    from oracle import frame_update as fu
    from paper_1806_04965_b200 import SrError
    g = graphs.dsr(2, batch=2, frames=4, h1_recurrence=False)
    X, Wt, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    want = fu.rollout_spec(g, "sequential", X, Wt, Bi)
    G = parity.make_graph(g, "sequential", "auto", 0, Wt, Bi)
    G.bind_window(2)
    x, o = parity.to_device(g, X[0]), G.output_node
    G.set_option(10, 0)
    G.reset([x[0]])
    G.rollout_window([x[1:3]])
    with pytest.raises(SrError) as e:
        G.sync_status()
    assert e.value.status == "SR_ERR_TIMEOUT"
    G.set_option(10, 1000)
    with pytest.raises(SrError):                        # recorded until the rollout starts over
        G.sync_status()
    G.reset([x[0]])
    out = torch.empty((4,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
    for t in (0, 2):
        G.rollout_window([x[t + 1:t + 3]], out[t:t + 2])
    G.sync_status()
    assert parity.rel_err(out.cpu().numpy().reshape(want[o][1:].shape), want[o][1:]) <= parity.TOL["bf16"]


@pytest.mark.parametrize("cin,k,stride,size", [(1, 1, 1, 9), (5, 5, 1, 11), (3, 3, 2, 10), (3, 3, 4, 32), (2, 7, 1, 8), (14, 3, 3, 13)])
def test_staged_input_edges(cin, k, stride, size):
    # receptive fields of 1 .. 126 values (filters are odd) (partial and full 16-byte chunks), windows that leave the image on every side,
    # odd sizes, strides; nine staged edges are more than one launch takes.  Half of them read the input inside the frame.
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    pad = (k - 1) // 2
    out = (size + 2 * pad - k) // stride + 1
    n = 9 if (cin, k) == (3, 3) else 2
    nodes = [Node("in", size, size, cin, IDENTITY)] + [Node("n%d" % i, out, out, 16) for i in range(n)] + [Node("o", 1, 1, 4, IDENTITY)]
    edges = [Edge(0, 1 + i, CONV, k, stride) for i in range(n)] + [Edge(1 + i, n + 1, GAP_DENSE) for i in range(min(n, 6))]
    g = GraphSpec("stems", nodes, edges, batch=3, frames=3, dtype="bf16", seed=91)
    check_shapes(g)
    g.patterns = {"p": [i % 2 for i in range(n)] + [1] * (len(edges) - n)}
    parity.check_stepwise(g, "p", zero_bias=False)
    parity.check_run(g, "p", graph_frames=2, resident=False)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,size,cin,c", [(3, 5, 3, 4), (3, 7, 8, 12), (2, 9, 60, 132), (130, 16, 4, 128)])
def test_cuda_core_convolutions_at_the_edges_of_their_tiles(batch, size, cin, c, dtype):
    # channel quads per block 1 .. 32 with a remainder, pixels that do not fill a block, reductions longer than the table in
    # shared memory (9 x 60 / 4 and 9 x 132 / 4 vectors, 25 x 3 scalars), one and (the last case) four pixels per thread
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    nodes = [Node("in", size, size, cin, IDENTITY), Node("a", size, size, c), Node("b", (size + 1) // 2, (size + 1) // 2, c, IDENTITY), Node("o", 1, 1, 3, IDENTITY)]
    edges = [Edge(0, 1, CONV, 5 if cin == 3 else 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 2), Edge(0, 2, CONV, 1, 2), Edge(2, 3, GAP_DENSE)]
    g = GraphSpec("tiles", nodes, edges, batch=batch, frames=2, dtype=dtype, seed=93)
    check_shapes(g)
    g.patterns = {"p": [1, 1, 1, 0, 1]}
    parity.check_stepwise(g, "p", engine="direct", zero_bias=False, samples=[0, batch - 1])


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_cuda_core_convolutions_of_images_with_a_million_rows(dtype):
    # one-dimensional signals of more than 2^20 samples, the last pixels of which do not fill a block; one and four pixels per thread
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    h = (1 << 20) + 37
    for stride, c in ((1, 4), (32, 8)):
        out = (h + stride - 1) // stride
        nodes = [Node("in", h, 1, 1, IDENTITY), Node("a", out, 1, c), Node("o", 1, 1, 2, IDENTITY)]
        g = GraphSpec("signal", nodes, [Edge(0, 1, CONV, 3, stride), Edge(1, 2, GAP_DENSE)], batch=1, frames=2, dtype=dtype, seed=95)
        check_shapes(g)
        g.patterns = {"p": [1, 1]}
        parity.check_stepwise(g, "p", engine="direct", zero_bias=False)


def test_cuda_core_convolution_of_a_sample_beyond_32_bit_offsets():
    # a source sample of 2^31 elements: the last rows and columns, which lie behind the middle of it, against a product made on the
    # GPU by torch in fp32 (the sums have four terms: 1e-2 is the rounding of the state to bf16, 2^-9, with room)
    import torch
    from paper_1806_04965_b200 import Graph
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, Node
    H, W, s = 1 << 15, 1 << 14, 64
    nodes = [Node("in", H, W, 4, IDENTITY), Node("a", H // s, W // s, 8, IDENTITY), Node("o", 1, 1, 2, IDENTITY)]
    G = Graph(nodes, [Edge(0, 1, CONV, 1, s), Edge(1, 2, GAP_DENSE)], [1, 1], batch=1, dtype="bf16", engine="direct")
    w = np.random.default_rng(4).standard_normal((8, 1, 1, 4)).astype(np.float32)
    G.set_weights([w, np.ones((2, 8), np.float32)], [np.zeros(n.c, np.float32) for n in nodes])
    x = torch.zeros((1, H, W, 4), dtype=torch.bfloat16, device="cuda:0")
    sub = torch.randn((H // s, W // s, 4), device="cuda:0", generator=torch.Generator(device="cuda:0").manual_seed(5)).to(torch.bfloat16)
    x[0, ::s, ::s] = sub
    G.reset([x])
    G.step([x])
    G.sync_status()
    want = torch.einsum("hwc,oc->hwo", sub.float(), torch.from_numpy(w.reshape(8, 4)).to("cuda:0").to(torch.bfloat16).float())
    got = G.get_state(1)[0].float()
    assert float((got - want).abs().max()) <= 1e-2 * float(want.abs().max())


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,size,cin,c", [(2, 5, 3, 4), (2, 7, 8, 132), (130, 16, 4, 64)])
def test_infinite_weights_leave_pixels_alone_whose_window_they_miss(batch, size, cin, c, dtype):
    # the weight of a corner tap is infinite: the first row and column, for which that tap lies outside the image, stay finite, with one
    # and (the last case) four pixels per thread; finite weights afterwards bring the usual results back
    import torch
    from oracle import frame_update as fu
    from workloads.graphs import CONV, GAP_DENSE, IDENTITY, Edge, GraphSpec, Node, check_shapes
    nodes = [Node("in", size, size, cin, IDENTITY), Node("a", size, size, c, IDENTITY), Node("o", 1, 1, 3, IDENTITY)]
    g = GraphSpec("inf", nodes, [Edge(0, 1, CONV, 3, 1), Edge(0, 1, CONV, 1, 1), Edge(1, 2, GAP_DENSE)], batch=batch, frames=1, dtype=dtype, seed=97)
    check_shapes(g)
    g.patterns = {"p": [1, 1, 1]}
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    bad = [w.copy() for w in W]
    bad[0][c - 1, 0, 0, cin - 1] = np.inf
    G = parity.make_graph(g, "p", "direct", 1, W, Bi)
    x = parity.to_device(g, X[0])
    samples = [0, batch - 1]
    for weights in (W, bad, W):
        with np.errstate(invalid="ignore"):
            want = fu.rollout_spec(g, "p", X, weights, Bi, samples=samples)[1][1]
        G.set_weights(weights)
        G.reset([x[0]])
        G.run([x[1:2]])                                 # (recorded in a CUDA graph)
        G.sync_status()
        got = G.get_state(1).float().cpu().numpy()[samples].reshape(want.shape)
        finite = np.isfinite(want)
        assert finite.all() == (weights is W) and np.array_equal(np.isfinite(got), finite)
        assert np.array_equal(got[~finite], want[~finite].astype(np.float32), equal_nan=True)
        assert parity.rel_err(got[finite], want[finite]) <= parity.TOL[dtype]
    # a pass that the caller recorded with finite weights keeps its kernel: pixels inside the image come out as they should
    out = torch.empty((1,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
    G.set_option(1, 0)
    stream, recorded = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.graph(recorded, stream=stream):
        G.reset([x[0]])
        G.run([x[1:2]], out)
    G.set_weights(bad)
    recorded.replay()
    torch.cuda.synchronize()
    with np.errstate(invalid="ignore"):
        want = fu.rollout_spec(g, "p", X, bad, Bi, samples=samples)[1][1]
    got = G.get_state(1).float().cpu().numpy()[samples].reshape(want.shape)
    inside = np.isfinite(want)
    inside[:, 0] = inside[:, :, 0] = False
    assert parity.rel_err(got[inside], want[inside]) <= parity.TOL[dtype]
    del recorded


@pytest.mark.parametrize("name,pattern", [("mini", "sequential"), ("mini", "mixed_input"), ("mini", "hybrid"), ("c3", "sequential"),
                                          ("c3", "hybrid"), ("dsr2", "sequential"), ("sink", "sequential")])
@pytest.mark.parametrize("graph_frames", [0, 2])
def test_frames_of_one_call_equal_calls_of_one_frame(name, pattern, graph_frames):
    # the input of a further frame of a call is queued beside the frame before it, where the pattern allows; every value is the same
    import torch
    spec = graphs.build(name, batch=2, frames=5)
    X, W, Bi = data.make_inputs(spec), data.make_weights(spec), data.make_biases(spec, zero=False)
    got = []
    for whole in (True, False):
        G = parity.make_graph(spec, pattern, "auto", graph_frames if whole else 0, W, Bi, resident=False)
        dev = {v: parity.to_device(spec, X[v]) for v in G.input_nodes}
        G.reset([dev[v][0] for v in G.input_nodes])
        out = torch.empty((5,) + tuple(G.out_shape()), dtype=torch.float32, device="cuda:0")
        if whole:
            G.run([dev[v][1:6] for v in G.input_nodes], out)
        else:
            for t in range(5):
                G.step([dev[v][t + 1] for v in G.input_nodes], out[t])
        G.sync_status()
        got.append([out] + [G.get_state(v) for v in range(len(spec.nodes))])
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,size,cin,c", [(1, 6, 16, 4), (20, 12, 16, 36), (40, 7, 24, 132), (3, 13, 14, 20)])
def test_cuda_core_convolutions_in_slices(batch, size, cin, c, dtype):
    # reductions of 128 values and more, which the warps of a block share: one and four pixels per thread, quads and pixels that do
    # not fill a block, several channel blocks, a source read value by value
    test_cuda_core_convolutions_at_the_edges_of_their_tiles(batch, size, cin, c, dtype)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch,size,cin,c", [(2, 7, 16, 132), (40, 7, 24, 132)])
def test_infinite_weights_on_items_whose_reduction_is_shared(batch, size, cin, c, dtype):
    # the warps of a block share the reduction; one and four pixels per thread
    test_infinite_weights_leave_pixels_alone_whose_window_they_miss(batch, size, cin, c, dtype)
