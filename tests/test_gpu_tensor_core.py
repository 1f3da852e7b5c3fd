"""GPU parity of the tcgen05 implicit-GEMM engine against the oracle: single edges of every kind the
engine lowers (taps, strides, channel-block widths, staged few-channel inputs, pooled edges, several
incoming edges), ragged tiles, and the reduced benchmark graphs with the engine chosen automatically."""
import pytest

from tests import parity
from workloads.graphs import CONV, GAP_DENSE, IDENTITY, RELU, Edge, GraphSpec, Node, check_shapes, build

pytestmark = pytest.mark.gpu


def tiny(name, nodes, edges, batch=3, frames=3, R=None):
    g = GraphSpec(name, nodes, edges, batch=batch, frames=frames, dtype="bf16", seed=4321)
    g.patterns = {"p": R or [1] * len(edges)}
    check_shapes(g)
    return g


def run(g):
    # as the library chooses; a work list per CTA instead of the shared list, on tiles of one lane of eight columns; tiles of four
    # lanes (or as many as the image is wide) with the shallowest weight ring
    from paper_1806_04965_b200 import Graph
    G = Graph(g.nodes, g.edges, g.patterns["p"], batch=g.batch, dtype="bf16")
    assert G.info["n_tensor_core_nodes"] >= 1, G.info
    parity.check_stepwise(g, "p", zero_bias=False, tc_lists=1, tile_width=8)
    parity.check_stepwise(g, "p", zero_bias=False, tile_width=32, weight_ring_units=2)
    return parity.check_stepwise(g, "p", zero_bias=False)


@pytest.mark.parametrize("cin,cout,k,stride,size", [
    (64, 64, 3, 1, 16), (64, 128, 3, 2, 16), (128, 256, 3, 4, 16), (64, 64, 1, 1, 16), (64, 128, 1, 2, 16),
    (32, 64, 3, 1, 16), (16, 32, 3, 1, 16), (48, 64, 3, 1, 8), (128, 128, 3, 8, 32), (64, 32, 3, 1, 28),
    (32, 64, 3, 2, 14), (32, 64, 3, 4, 28), (256, 256, 3, 1, 8), (64, 96, 3, 1, 7),
])
def test_single_conv_edge(cin, cout, k, stride, size):
    out = size // stride
    for R in ([0], [1]):
        g = tiny("edge", [Node("in", size, size, cin, IDENTITY), Node("n", out, out, cout, RELU), Node("o", 1, 1, 4, IDENTITY)],
                 [Edge(0, 1, CONV, k, stride), Edge(1, 2, GAP_DENSE)], R=R + [1])
        run(g)


def test_few_channel_input_edges_are_staged():
    for cin, k in ((3, 3), (1, 3), (3, 1)):
        g = tiny("stem", [Node("in", 16, 16, cin, IDENTITY), Node("a", 16, 16, 64), Node("b", 16, 16, 64),
                          Node("o", 1, 1, 4, IDENTITY)],
                 [Edge(0, 1, CONV, k, 1), Edge(1, 2, CONV, 3, 1), Edge(0, 2, CONV, k, 1), Edge(1, 1, CONV, 3, 1),
                  Edge(2, 3, GAP_DENSE)], frames=4, R=[1, 1, 0, 1, 0])
        run(g)
        for ring in (3, 8):
            parity.check_stepwise(g, "p", zero_bias=False, weight_ring_units=ring)


def test_a_node_fed_by_a_staged_edge_only():
    # no tap of node a shares an activation box: flat tiles (0), or tiles of lanes where a width is asked for
    g = tiny("stem_only", [Node("in", 32, 32, 3, IDENTITY), Node("a", 32, 32, 64), Node("b", 32, 32, 128), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)], batch=5, frames=4)
    for tile_width in (0, 8, 32):
        parity.check_stepwise(g, "p", zero_bias=False, tile_width=tile_width)


@pytest.mark.parametrize("c,act_b", [(64, RELU), (32, IDENTITY)])
def test_two_narrow_nodes_that_share_a_source_run_as_one_plan(c, act_b):
    # a <- {in (staged), a}, b <- {a, b, in (1x1, staged)}, d <- {a, b}: a and b have the same shape, at most 64 channels
    # and both read a through a 3x3 filter from the previous frame, so b's weights take rows 64..127 of a's tiles
    g = tiny("fused", [Node("in", 24, 16, 3, IDENTITY), Node("a", 24, 16, c), Node("b", 24, 16, c, act_b), Node("d", 12, 8, 128),
                       Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(2, 2, CONV, 3, 1), Edge(0, 2, CONV, 1, 1),
              Edge(1, 3, CONV, 3, 2), Edge(2, 3, CONV, 1, 2), Edge(3, 4, GAP_DENSE)], batch=5, frames=4)
    for fuse in (1, 0):
        parity.check_stepwise(g, "p", zero_bias=False, tc_fuse=fuse)
    parity.check_stepwise(g, "p", zero_bias=False, tc_fuse=1, tc_lists=1, weight_ring_units=2)
    # with a -> b inside the frame (R = 0) the two nodes are in different launch groups: nothing to fuse, same results
    g.patterns["q"] = [1, 1, 0, 1, 1, 1, 1, 1]
    parity.check_stepwise(g, "q", zero_bias=False)


def test_pooled_edge_and_recurrence():
    g = tiny("pool", [Node("in", 16, 16, 64, IDENTITY), Node("a", 8, 8, 128), Node("b", 8, 8, 128), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1, 2), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(0, 2, CONV, 3, 2),
              Edge(2, 3, GAP_DENSE)], frames=4)
    run(g)


def test_rectangular_images_and_odd_batch():
    g = tiny("rect", [Node("in", 12, 20, 64, IDENTITY), Node("a", 12, 20, 64), Node("b", 6, 10, 64),
                      Node("o", 1, 1, 5, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 2), Edge(2, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)],
             batch=5, frames=4)
    run(g)


@pytest.mark.parametrize("name,kw", [
    ("c2", dict(batch=3, frames=6)),
    ("c3", dict(batch=2, frames=4, size=16)),
    ("c3", dict(batch=5, frames=3, size=32)),
    ("c4", dict(batch=2, frames=4, size=16)),
    ("c5", dict(batch=2, frames=4, size=16)),
])
def test_configs_reduced_tensor_cores(name, kw):
    g = build(name, **kw)
    for p in g.patterns:
        parity.check_stepwise(g, p, engine="auto", zero_bias=False)
        parity.check_stepwise(g, p, engine="auto", zero_bias=False, tile_width=32)
        parity.check_run(g, p, engine="auto", graph_frames=2)
        parity.check_run(g, p, engine="auto", graph_frames=2, tile_width=16, resident=False)


@pytest.mark.parametrize("batch", [1, 2, 7])
def test_lanes_with_ragged_batches_and_widths(batch):
    # the last lanes of a tile lie partly or wholly outside the image (20, 10 and 5 columns in lanes of eight)
    g = tiny("ragged", [Node("in", 20, 20, 64, IDENTITY), Node("a", 20, 20, 128), Node("b", 10, 10, 128), Node("c", 5, 5, 256),
                        Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 2), Edge(2, 2, CONV, 3, 1), Edge(2, 3, CONV, 3, 2),
              Edge(0, 3, CONV, 1, 4), Edge(3, 4, GAP_DENSE)], batch=batch, frames=3)
    run(g)


@pytest.mark.parametrize("k", [0, 2, 6])
def test_paper_cifar10_networks_on_tensor_cores(k):
    # DSR0 / DSR2 / DSR6 (Sec. A, paragraph CIFAR10): receptive field 5 on the 3-channel input (75 columns, staged as two
    # K-blocks), 32- and 64-channel blocks with dense skips, stride-4 edges into the 4 x 4 x 512 node (four channel
    # tiles); every convolutional node runs on the tensor cores, only the dense output node does not
    from paper_1806_04965_b200 import Graph
    from workloads import graphs
    g = graphs.dsr(k, batch=3, frames=4)
    G = Graph(g.nodes, g.edges, g.patterns["streaming"], batch=g.batch, dtype="bf16")
    assert G.info["n_direct_nodes"] == 1 and G.info["n_tensor_core_nodes"] == len(g.nodes) - 2, G.info
    assert G.info["first_response_step"] == 4
    S = Graph(g.nodes, g.edges, g.patterns["sequential"], batch=0)
    assert S.info["first_response_step"] == 4 + k and S.info["inference_factor"] == 4 + k
    for p in g.patterns:
        parity.check_stepwise(g, p, zero_bias=False)
        parity.check_stepwise(g, p, zero_bias=False, tile_width=16)
        parity.check_run(g, p, graph_frames=2)


def test_gtsrb_network_variant():
    # DSR4 without the H1 recurrence and with 43 classes (Sec. A, paragraph GTSRB)
    from workloads import graphs
    g = graphs.dsr(4, batch=2, frames=3, classes=43, h1_recurrence=False)
    parity.check_stepwise(g, "streaming", zero_bias=False)


@pytest.mark.parametrize("tile_width,ring", [(0, 0), (8, 0), (16, 4), (32, 3), (32, 8)])
@pytest.mark.parametrize("size", [(9, 5), (7, 17), (5, 33), (3, 70)])
def test_tile_widths_and_ring_depths(size, tile_width, ring):
    # a width of 8, 16 or 32 makes tiles of one, two or four lanes of eight columns, as far as the image is wide, the last of them
    # beyond it; blocks of 64, 32 and 16 channels and a staged edge in one reduction, which make bursts of two weight groups and of one
    h, w = size
    g = tiny("lanes", [Node("in", h, w, 3, IDENTITY), Node("a", h, w, 64), Node("b", h, w, 48), Node("c", h, w, 96), Node("d", (h + 1) // 2, (w + 1) // 2, 136),
                       Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(0, 2, CONV, 1, 1), Edge(2, 3, CONV, 3, 1), Edge(1, 3, CONV, 1, 1),
              Edge(3, 3, CONV, 3, 1), Edge(3, 4, CONV, 3, 2), Edge(2, 4, CONV, 1, 2), Edge(4, 5, GAP_DENSE)], batch=3, frames=3)
    parity.check_stepwise(g, "p", zero_bias=False, tile_width=tile_width, weight_ring_units=ring)


@pytest.mark.parametrize("h,w", [(1, 250), (2, 131), (1, 20001), (4, 20001)])
def test_images_of_few_rows(h, w):
    # tiles of as many lanes as an accumulator holds: four of 16 columns, two, eight of 16 and eight of 32 (a lane has at least 16
    # columns, of which one row of eight pixels fills half)
    g = tiny("rows", [Node("in", h, w, 64, IDENTITY), Node("a", h, w, 64), Node("b", h, w, 32), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)], batch=1, frames=2)
    parity.check_stepwise(g, "p", zero_bias=False)


@pytest.mark.parametrize("name,kw", [("c3", dict(batch=3, frames=4, size=16)), ("c4", dict(batch=2, frames=4, size=16)), ("dsr2", dict(batch=2, frames=3)),
                                     ("c2", dict(batch=2, frames=4, dtype="fp32")), ("mini", dict(batch=2, frames=4, dtype="fp32"))])
def test_launches_one_after_the_other_give_the_same(name, kw):
    # overlap off (option 4): every launch waits for the one before it; the same kernels on the same data, bit for bit, also recorded
    # in CUDA graphs
    import torch
    from workloads import data, graphs
    g = graphs.dsr(2, **kw) if name == "dsr2" else build(name, **kw)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    for p in g.patterns:
        seen = []
        for overlap, graph_frames in ((1, 0), (0, 0), (0, 2), (1, 2)):
            G = parity.make_graph(g, p, "auto", graph_frames, W, Bi, resident=False)
            G.set_option(4, overlap)
            out = G.rollout([parity.to_device(g, X[v]) for v in G.input_nodes])
            G.sync_status()
            seen.append([out] + [G.get_state(v) for v in range(len(g.nodes))])
        for other in seen[1:]:
            assert all(torch.equal(a, b) for a, b in zip(seen[0], other)), p
        parity.check_run(g, p, resident=False)


def test_a_state_of_more_than_2_31_elements():
    # 514 samples of 128 x 128 x 256: the last samples lie beyond 32-bit element offsets; first and last ones against the oracle
    import numpy as np
    from oracle import frame_update as fu
    from workloads import data
    g = tiny("large", [Node("in", 128, 128, 1, IDENTITY), Node("a", 128, 128, 256), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 2, GAP_DENSE)], batch=514, frames=2)
    assert g.batch * 128 * 128 * 256 > 1 << 31
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    samples = [0, 511, 512, 513]
    want = fu.rollout_spec(g, "p", X, W, Bi, samples=samples)
    G = parity.make_graph(g, "p", "auto", 0, W, Bi)
    assert G.info["n_tensor_core_nodes"] == 1
    out = G.rollout([parity.to_device(g, X[0])])
    G.sync_status()
    assert parity.rel_err(out.cpu().numpy()[:, samples].reshape(want[2][1:].shape), want[2][1:]) <= parity.TOL["bf16"]
    state = G.get_state(1)
    for i, b in enumerate(samples):
        assert parity.rel_err(state[b].float().cpu().numpy(), want[1][2][i]) <= parity.TOL["bf16"], b


@pytest.mark.parametrize("name,kw", [("c3", dict(batch=40, frames=2, size=16)), ("c4", dict(batch=3, frames=2, size=16))])
def test_the_wait_limit_does_not_count_the_run_before(name, kw):
    # a launch that starts early, beside a run of another graph that takes far longer (4000 frames of the resident kernel, some 15 ms)
    # than the limit of its own waits (1 ms); c4 has more nodes than a CTA keeps tables, c3 several work items per CTA
    import torch
    from oracle import frame_update as fu
    from workloads import data
    long = build("c2", batch=8, frames=1)
    L = parity.make_graph(long, "streaming", "auto", 0, data.make_weights(long), data.make_biases(long))
    assert L.info["resident_cluster"] > 0
    xl = torch.zeros((4001, 8, 28, 28, 1), dtype=torch.bfloat16, device="cuda:0")
    g = build(name, **kw)
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    samples = [0, g.batch - 1]
    want = fu.rollout_spec(g, "streaming", X, W, Bi, samples=samples)
    G = parity.make_graph(g, "streaming", "auto", 0, W, Bi, wait_limit_ms=1)
    x, o = parity.to_device(g, X[0]), G.output_node
    out = torch.empty((2,) + G.out_shape(), dtype=torch.float32, device="cuda:0")
    L.reset([xl[0]])
    G.reset([x[0]])
    for t in (1, 2):
        L.run([xl[1:]])
        G.step([x[t]], out[t - 1])
        G.sync_status()
    assert parity.rel_err(out.cpu().numpy()[:, samples].reshape(want[o][1:].shape), want[o][1:]) <= parity.TOL["bf16"]


@pytest.mark.parametrize("cin,c,k,stride,size,batch", [
    (256, 256, 3, 1, 8, 1),        # two edges of 36 K-blocks on one tile of 64 pixels
    (256, 128, 3, 1, 8, 5),
    (48, 96, 3, 1, 7, 2),          # 16-channel K-blocks, channels and pixels that fill no tile
    (64, 512, 3, 4, 16, 1),        # a box per tap; 16 pixels: parts without columns of their own
    (128, 64, 3, 2, 28, 37),       # wide tiles, their sums in the rings
    (64, 128, 1, 1, 12, 1),        # one K-block per edge: nothing to cut
])
def test_long_reductions_of_few_pixels(cin, c, k, stride, size, batch):
    # launches with fewer items than SMs, whose items are cut along K over the CTAs of a cluster
    out = size // stride
    g = tiny("split", [Node("in", size, size, cin, IDENTITY), Node("a", out, out, c), Node("b", out, out, c), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, k, stride), Edge(1, 1, CONV, k, 1), Edge(1, 2, CONV, k, 1), Edge(2, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)],
             batch=batch, frames=3)
    samples = list(range(min(batch, 4))) + ([batch - 1] if batch > 4 else [])
    parity.check_stepwise(g, "p", samples=samples, zero_bias=False)
    g.patterns["q"] = [0, 1, 0, 1, 0]
    parity.check_stepwise(g, "q", samples=samples, zero_bias=False)


@pytest.mark.parametrize("c,size,batch", [
    (256, 8, 127),                 # two images to a tile, the last one alone
    (256, 8, 25),                  # the same with the reduction cut: nine chunks of columns do not divide by the parts
    (256, 5, 60),                  # three images, all 160 columns; the parts' sums in the rings
])
def test_tiles_of_a_few_small_images(c, size, batch):
    g = tiny("pair", [Node("in", size, size, 64, IDENTITY), Node("a", size, size, c), Node("b", size, size, c), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)], batch=batch, frames=3)
    g.patterns["q"] = [0, 1, 0, 0]
    for pattern in ("p", "q"):
        parity.check_stepwise(g, pattern, samples=[0, 1, 2, batch // 2, batch - 2, batch - 1], zero_bias=False)


@pytest.mark.parametrize("c,n", [(32, 3), (32, 4), (32, 5), (64, 3)])
def test_several_narrow_nodes_that_share_sources(c, n):
    # a block in which every earlier node feeds every later one, as in the paper's CIFAR10 networks: up to 128 channels run as one
    # plan; the nodes' activations and biases stay their own, the last plan may be part empty
    nodes = [Node("in", 12, 20, 3, IDENTITY)] + [Node("n%d" % i, 12, 20, c, IDENTITY if i == 1 else RELU) for i in range(n)]
    edges = [Edge(0, 1, CONV, 5, 1), Edge(1, 1, CONV, 3, 1)] + [Edge(i, j, CONV, 3, 1) for i in range(1, n + 1) for j in range(i + 1, n + 1)]
    g = tiny("block", nodes + [Node("o", 1, 1, 4, IDENTITY)], edges + [Edge(i, n + 1, GAP_DENSE) for i in range(1, n + 1)], batch=3, frames=4)
    for fuse in (1, 0):
        parity.check_stepwise(g, "p", zero_bias=False, tc_fuse=fuse)
    parity.check_stepwise(g, "p", zero_bias=False, tc_lists=1, weight_ring_units=2, tile_width=16)


def plans(g, pattern, **options):
    """How the launch groups of a pattern are planned: the path that a case means to take."""
    from paper_1806_04965_b200 import Graph
    G = Graph(g.nodes, g.edges, g.patterns[pattern], batch=g.batch, dtype="bf16", **options)
    return [G.launch_plan(i) for i in range(G.info["n_groups"])]


@pytest.mark.parametrize("cin,c,k,stride,size,batch,parts,rings,columns", [
    (256, 256, 3, 1, 8, 1, 8, 0, 64),
    (256, 128, 3, 1, 8, 5, 8, 0, 64),
    (48, 96, 3, 1, 7, 2, 8, 0, 64),
    (64, 512, 3, 4, 16, 1, 8, 0, 32),          # two chunks of columns: parts without columns of their own
    (128, 64, 3, 2, 28, 37, 2, 0, 112),        # two nodes to a plan
    (128, 256, 3, 1, 8, 12, 4, 1, 144),        # sums in the rings, nine chunks of columns over four parts
    (64, 256, 3, 1, 16, 20, 2, 1, 256),        # sums in the rings, the widest tile
    (64, 128, 1, 1, 12, 1, 8, 0, 64),          # one K-block per 1 x 1 edge (in the second pattern a launch with nothing to cut)
])
def test_long_reductions_take_the_path_that_is_meant(cin, c, k, stride, size, batch, parts, rings, columns):
    out = size // stride
    g = tiny("split", [Node("in", size, size, cin, IDENTITY), Node("a", out, out, c), Node("b", out, out, c), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, k, stride), Edge(1, 1, CONV, k, 1), Edge(1, 2, CONV, k, 1), Edge(2, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)],
             batch=batch, frames=3)
    plan = plans(g, "p")[0]
    assert (plan["parts"], plan["sums_in_rings"], plan["columns"]) == (parts, rings, columns), plan
    if k == 1:
        g.patterns["q"] = [0, 1, 0, 1, 0]
        assert plans(g, "q")[0]["parts"] == 1
    if rings:
        test_long_reductions_of_few_pixels(cin, c, k, stride, size, batch)


@pytest.mark.parametrize("c,size,batch,parts,rings,columns", [
    (256, 8, 127, 1, 0, 144),
    (256, 8, 25, 2, 0, 144),
    (256, 5, 60, 2, 1, 208),       # four images to a tile
])
def test_tiles_of_a_few_small_images_take_the_path_that_is_meant(c, size, batch, parts, rings, columns):
    g = tiny("pair", [Node("in", size, size, 64, IDENTITY), Node("a", size, size, c), Node("b", size, size, c), Node("o", 1, 1, 4, IDENTITY)],
             [Edge(0, 1, CONV, 3, 1), Edge(1, 1, CONV, 3, 1), Edge(1, 2, CONV, 3, 1), Edge(2, 3, GAP_DENSE)], batch=batch, frames=3)
    plan = plans(g, "p")[0]
    assert (plan["parts"], plan["sums_in_rings"], plan["columns"]) == (parts, rings, columns), plan


@pytest.mark.parametrize("c,n,joined", [(32, 3, 2), (32, 4, 4), (32, 5, 2), (64, 3, 2)])
def test_narrow_nodes_that_share_sources_are_joined(c, n, joined):
    nodes = [Node("in", 12, 20, 3, IDENTITY)] + [Node("n%d" % i, 12, 20, c, IDENTITY if i == 1 else RELU) for i in range(n)]
    edges = [Edge(0, 1, CONV, 5, 1), Edge(1, 1, CONV, 3, 1)] + [Edge(i, j, CONV, 3, 1) for i in range(1, n + 1) for j in range(i + 1, n + 1)]
    g = tiny("block", nodes + [Node("o", 1, 1, 4, IDENTITY)], edges + [Edge(i, n + 1, GAP_DENSE) for i in range(1, n + 1)], batch=3, frames=4)
    for fuse in (1, 0):
        assert plans(g, "p", tc_fuse=fuse)[0]["joined"] == (joined if fuse else 1)


@pytest.mark.parametrize("c,n,cin,size,batch,joined,parts", [
    (32, 4, 64, 12, 2, 4, 8),              # few items: the reduction is cut, parts without K-blocks for some of the nodes
    (32, 4, 64, 16, 160, 2, 1),            # many items
    (32, 3, 16, 12, 40, 3, 1),             # rows without a node; K-blocks of 16 channels
    (64, 2, 32, 16, 3, 2, 8),
    (64, 2, 128, 28, 37, 2, 1),
])
def test_an_infinity_stays_with_the_nodes_that_read_it(c, n, cin, size, batch, joined, parts):
    # nodes that share a source run as one plan; what only one of them reads must not reach the others, at any pixel, whether the first
    # K-blocks of the plan serve all nodes or not
    import numpy as np
    import torch
    from oracle import frame_update as fu
    from workloads import data
    nodes = [Node("x", size, size, 48, IDENTITY), Node("y", size, size, cin, IDENTITY)]
    nodes += [Node("n%d" % i, size, size, c, RELU if i else IDENTITY) for i in range(n)] + [Node("o", 1, 1, 4, IDENTITY)]
    edges = [Edge(0, 2 + i, CONV, 3, 1) for i in range(n)] + [Edge(1, 2, CONV, 3, 1)]
    edges += [Edge(2 + i, 2 + i, CONV, 3, 1) for i in range(n)] + [Edge(1 + n, 2 + n, GAP_DENSE)]
    g = tiny("inf", nodes, edges, batch=batch, frames=3)
    plan = plans(g, "p")[0]
    assert (plan["joined"], plan["parts"], plan["masked"]) == (joined, parts, 1), plan
    samples = [0, batch // 2, batch - 1]
    X, W, Bi = data.make_inputs(g), data.make_weights(g), data.make_biases(g, zero=False)
    X[1][0, :, 1, 1, :] = np.inf
    X[1][1, :, size - 1, 2, 0] = -np.inf
    want = fu.rollout_spec(g, "p", X, W, Bi, samples=samples)
    for options in ({}, {"tile_width": 32, "weight_ring_units": 2}, {"tile_width": 8}):
        G = parity.make_graph(g, "p", "auto", 0, W, Bi, **options)
        dev = [parity.to_device(g, X[v]) for v in (0, 1)]
        G.reset([d[0] for d in dev])
        for t in range(1, 4):
            G.step([d[t] for d in dev], None)
            for v in range(2, 2 + n):
                got = G.get_state(v).float().cpu().numpy()[samples]
                finite = np.isfinite(want[v][t])
                assert finite.all() == (v > 2)
                assert np.abs(got[finite] - want[v][t][finite]).max() <= parity.TOL["bf16"] * np.abs(want[v][t][finite]).max(), (options, v, t)
        G.sync_status()
