"""Parity of the TreeRNN and RNTN forward (the paper's other two evaluation models, Section 6.1)
through the C ABI against their fp64 oracle: schedule bit-exact, states within 1e-4 max-abs (fp32
arithmetic) and within 1e-4 of the largest state."""
import numpy as np
import pytest
import torch

from oracle import recursive_cells_oracle as rc
from oracle import treelstm_oracle as orc
from paper_1809_00832_b200 import binding, forests as fg
from tests import util

pytestmark = pytest.mark.gpu

MODES = [binding.PER_LEVEL, binding.PERSISTENT]
KIND = {binding.CELL_TREERNN: rc.TREERNN, binding.CELL_RNTN: rc.RNTN}


def _model(cell, p):
    util.lib_ready()
    V = util.to_dev(p.V) if p.V is not None else None
    return binding.TreeLSTM.recursive(cell, p.H, p.vocab, util.to_dev(p.emb), util.to_dev(p.W), util.to_dev(p.b), V)


def _check(cell, p, forest, flags):
    model = _model(cell, p)
    res = util.gpu_forward(model, forest, flags)
    status, _, level, order, off = orc.schedule(forest.left, forest.right)
    util.check_schedule(res, dict(level=level, order=order, level_offset=off), forest.n_nodes)
    h = rc.forward_recursive(KIND[cell], forest.left, forest.right, forest.token, p.emb, p.W, p.b, p.V)
    err = util.max_abs(res["h"], h)
    assert err < util.TOL["fp32"], err
    assert err <= 1e-4 * np.max(np.abs(h))
    assert "c" not in res                               # these cells have no cell state
    np.testing.assert_array_equal(res["h"][forest.left < 0], p.emb[forest.token[forest.left < 0]])
    return model, res, h


@pytest.mark.parametrize("flags", MODES)
@pytest.mark.parametrize("H", [16, 50, 150])
def test_treernn_matches_oracle(H, flags):
    """sizes below, across and above one 64-unit tile; several row tiles and a ragged tail; permuted ids"""
    rng = np.random.default_rng(100 + H)
    p = fg.draw_recursive_params(rng, H, 300, tensor=False, emb_scale=0.8, w_scale=1.5 / np.sqrt(2 * H))
    forest = fg.random_forest(rng, 25, 2, 56, 300)
    forest, _ = fg.permute_node_ids(forest, rng)
    _check(binding.CELL_TREERNN, p, forest, flags)


@pytest.mark.parametrize("flags", MODES)
@pytest.mark.parametrize("H", [8, 25, 40])
def test_rntn_matches_oracle(H, flags):
    """the tensor term is a contraction over 4H^2 products per node; H = 25 (the size of the original
    model) and sizes that match no tile"""
    rng = np.random.default_rng(200 + H)
    p = fg.draw_recursive_params(rng, H, 200, tensor=True, emb_scale=0.8, w_scale=1.0 / np.sqrt(2 * H),
                                 v_scale=1.0 / (2 * H))
    forest = fg.random_forest(rng, 12, 1, 30, 200)
    forest, _ = fg.permute_node_ids(forest, rng)
    model, res, h = _check(binding.CELL_RNTN, p, forest, flags)
    # the tensor term matters at these scales: the same forest without it differs visibly
    h0 = rc.forward_recursive(rc.TREERNN, forest.left, forest.right, forest.token, p.emb, p.W, p.b)
    assert np.max(np.abs(h0 - h)) > 50 * util.TOL["fp32"]


@pytest.mark.parametrize("cell", [binding.CELL_TREERNN, binding.CELL_RNTN])
def test_shape_extremes_edge_cases_and_roots(cell):
    """left chains (one node per tree and wavefront), balanced trees, single leaves, the empty forest;
    roots come back with their states"""
    rng = np.random.default_rng(7)
    H = 24
    p = fg.draw_recursive_params(rng, H, 50, tensor=cell == binding.CELL_RNTN, emb_scale=0.8,
                                 w_scale=1.0 / np.sqrt(2 * H), v_scale=1.0 / (2 * H))
    shapes = [fg.left_chain_shape(40), fg.balanced_shape(64), None, None, fg.left_chain_shape(3)]
    forest = fg.forest_from_shapes(shapes, rng, 50)
    for flags in MODES:
        model, res, h = _check(cell, p, forest, flags)
        assert res["n_levels"] == 40
        roots = model.roots(forest.n_trees)
        torch.cuda.synchronize()
        ids = roots["root_ids"].cpu().numpy()
        np.testing.assert_array_equal(ids, np.sort(forest.roots))
        np.testing.assert_array_equal(roots["root_h"].cpu().numpy(), res["h"][ids])
    empty = fg.Forest(*(np.zeros(0, dtype=np.int32) for _ in range(5)))
    model = _model(cell, p)
    for flags in MODES:
        assert util.gpu_forward(model, empty, flags)["n_levels"] == 0
    # a malformed forest is still an error code; a backward without a classifier is refused
    bad = [torch.tensor(x, dtype=torch.int32, device="cuda") for x in ([-1, -1, 0], [-1, -1, 3], [0, 1, -1])]
    with pytest.raises(binding.TreeLSTMError) as err:
        model.forward(*bad, flags=binding.PERSISTENT)
    assert err.value.code == binding.ERR_INVALID_FOREST
    good = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
    model.forward(*good, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    with pytest.raises(binding.TreeLSTMError) as err:
        model.backward_recursive(util.to_dev(np.zeros(forest.n_nodes, np.int32)), forest.n_leaves)
    assert err.value.code in (binding.ERR_STATE, binding.ERR_INVALID_ARG)    # no classifier: empty gradient buffers


def test_treernn_large_hidden_size_and_host_entry_point():
    """H = 256 (four unit tiles, 64 KB of staged child states per tile) through the host-buffer call"""
    rng = np.random.default_rng(9)
    H = 256
    p = fg.draw_recursive_params(rng, H, 400, tensor=False, emb_scale=0.8, w_scale=1.5 / np.sqrt(2 * H))
    forest = fg.random_forest(rng, 30, 2, 56, 400)
    model = _model(binding.CELL_TREERNN, p)
    host = binding.pack_forest_host(forest.left, forest.right, forest.token)
    out = model.forward_host(*host, all_states=True, max_roots=forest.n_trees)
    h = rc.forward_recursive(rc.TREERNN, forest.left, forest.right, forest.token, p.emb, p.W, p.b)
    assert util.max_abs(out["h"].numpy(), h) < util.TOL["fp32"]
    roots = np.sort(forest.roots)
    np.testing.assert_array_equal(out["root_ids"].numpy(), roots)
    assert util.max_abs(out["root_h"].numpy(), h[roots]) < util.TOL["fp32"]


def _training_step(cell, p, forest, flags, n_classes=5, seed=7):
    rng = np.random.default_rng(seed)
    Wc = rng.uniform(-0.3, 0.3, size=(p.H, n_classes)).astype(np.float32)
    bc = rng.uniform(-0.1, 0.1, size=n_classes).astype(np.float32)
    labels = rng.integers(0, n_classes, size=forest.n_nodes).astype(np.int32)
    ref = rc.loss_and_gradients(KIND[cell], forest.left, forest.right, forest.token, p.emb, p.W, p.b, Wc, bc, labels, p.V)
    model = _model(cell, p)
    model.set_classifier(util.to_dev(Wc), util.to_dev(bc))
    model.forward(util.to_dev(forest.left), util.to_dev(forest.right), util.to_dev(forest.token),
                  flags=flags | binding.SAVE_FOR_BACKWARD)
    g = {k: v.cpu().numpy() for k, v in model.backward_recursive(util.to_dev(labels), forest.n_leaves).items()}
    util.compare_training_step(g, ref, util.TOL["fp32"], util.REL["fp32"], loss_rel=1e-5)
    if cell == binding.CELL_RNTN:
        err, scale = util.max_abs(g["dV"], ref["dV"]), float(np.max(np.abs(ref["dV"])))
        assert err < util.TOL["fp32"] and err <= util.REL["fp32"] * scale, (err, scale)
        assert scale > 0 or forest.n_nodes == forest.n_leaves
    model.close()
    return g, ref


@pytest.mark.parametrize("flags", MODES)
@pytest.mark.parametrize("H", [16, 50, 130])
def test_treernn_training_step_matches_oracle(H, flags):
    """loss and every gradient group (dW, db, dWc, dbc, touched embedding rows) of backpropagation
    through structure against the fp64 oracle: absolute 1e-4 and 2e-5 of each group's largest entry;
    duplicate tokens (vocabulary smaller than the number of leaves) accumulate into one row"""
    rng = np.random.default_rng(300 + H)
    p = fg.draw_recursive_params(rng, H, 40, tensor=False, emb_scale=0.8, w_scale=1.5 / np.sqrt(2 * H))
    forest = fg.random_forest(rng, 20, 1, 40, 40)
    forest, _ = fg.permute_node_ids(forest, rng)
    g, ref = _training_step(binding.CELL_TREERNN, p, forest, flags)
    assert len(ref["touched_ids"]) < forest.n_leaves          # duplicates were there
    assert float(np.max(np.abs(ref["dW"]))) > 100 * util.TOL["fp32"] * util.REL["fp32"]


@pytest.mark.parametrize("flags", MODES)
@pytest.mark.parametrize("H", [8, 25])
def test_rntn_training_step_matches_oracle(H, flags):
    """the same with the tensor term: dV [H][2H][2H] and the (V_j + V_j^T) x part of the children's gradient"""
    rng = np.random.default_rng(400 + H)
    p = fg.draw_recursive_params(rng, H, 60, tensor=True, emb_scale=0.8, w_scale=1.0 / np.sqrt(2 * H),
                                 v_scale=1.0 / (2 * H))
    forest = fg.random_forest(rng, 10, 1, 24, 60)
    forest, _ = fg.permute_node_ids(forest, rng)
    _training_step(binding.CELL_RNTN, p, forest, flags)


def test_recursive_training_edge_cases():
    """a forest of single-leaf trees only (no internal node: dW, db, dV are zero, the embedding rows carry
    the classifier's gradient), and the wrong backward call for the context kind is refused"""
    rng = np.random.default_rng(500)
    p = fg.draw_recursive_params(rng, 12, 30, tensor=True, emb_scale=0.8, w_scale=0.3, v_scale=0.05)
    forest = fg.random_forest(rng, 9, 1, 1, 30)
    g, ref = _training_step(binding.CELL_RNTN, p, forest, binding.PERSISTENT)
    assert not g["dW"].any() and not g["dV"].any() and not g["db"].any()
    model = _model(binding.CELL_TREERNN, p)
    model.set_classifier(util.to_dev(np.zeros((12, 3), np.float32)), util.to_dev(np.zeros(3, np.float32)))
    model.forward(util.to_dev(forest.left), util.to_dev(forest.right), util.to_dev(forest.token),
                  flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    with pytest.raises(binding.TreeLSTMError):
        model.backward(util.to_dev(np.zeros(forest.n_nodes, np.int32)), forest.n_leaves)
    model.close()


@pytest.mark.parametrize("cell,H,n_trees,hi", [
    (binding.CELL_TREERNN, 63, 9, 40), (binding.CELL_TREERNN, 64, 9, 40), (binding.CELL_TREERNN, 254, 6, 30), (binding.CELL_TREERNN, 257, 6, 30),
    (binding.CELL_TREERNN, 128, 300, 12), (binding.CELL_RNTN, 1, 5, 9), (binding.CELL_RNTN, 32, 60, 20), (binding.CELL_RNTN, 33, 5, 20)])
def test_training_step_at_the_limits_of_the_tree_kernels(cell, H, n_trees, hi):
    """sizes at which the cluster grows and at which the tree kernels end; more trees than clusters; a depth wider
    than a pass; single leaves and chains among the trees"""
    rng = np.random.default_rng(600 + H)
    tensor = cell == binding.CELL_RNTN
    p = fg.draw_recursive_params(rng, H, 90, tensor=tensor, emb_scale=0.8, w_scale=1.0 / np.sqrt(2 * H), v_scale=1.0 / (2 * H))
    forest = fg.concat_forests([fg.random_forest(rng, n_trees, 1, hi, 90),
                                fg.forest_from_shapes([fg.left_chain_shape(17), fg.balanced_shape(32)], rng, 90)])
    _training_step(cell, p, forest, binding.PERSISTENT)


def test_states_that_do_not_fit_shared_memory():
    """two trees of a thousand leaves each: the states of a cluster go through L2"""
    rng = np.random.default_rng(700)
    p = fg.draw_recursive_params(rng, 130, 90, tensor=False, emb_scale=0.8, w_scale=1.0 / np.sqrt(260))
    forest = fg.random_forest(rng, 2, 1000, 1001, 90)
    _training_step(binding.CELL_TREERNN, p, forest, binding.PERSISTENT)


LARGE = {"few large trees": lambda rng: [fg.balanced_shape(1024)] + [fg.random_split_shape(rng, 9) for _ in range(7)] + [None],
         "one chain": lambda rng: [fg.left_chain_shape(900)],
         "many trees": lambda rng: [fg.random_split_shape(rng, int(n)) for n in rng.integers(1, 30, size=120)],
         "tables that fill shared memory": lambda rng: [fg.random_split_shape(rng, int(n)) for n in rng.integers(2, 56, size=310)]}


@pytest.mark.parametrize("kind", LARGE)
@pytest.mark.parametrize("cell,H", [(binding.CELL_TREERNN, 20), (binding.CELL_TREERNN, 130), (binding.CELL_RNTN, 8)])
def test_large_forests_on_either_way(cell, H, kind):
    """forests beyond those that always go to the clusters: the tree kernel leaves some of them to the kernels that take a
    wavefront over the whole GPU, forward and backward, and walks the others, from a sample of their nodes"""
    rng = np.random.default_rng(900 + H)
    tensor = cell == binding.CELL_RNTN
    p = fg.draw_recursive_params(rng, H, 90, tensor=tensor, emb_scale=0.8, w_scale=1.0 / np.sqrt(2 * H), v_scale=1.0 / (2 * H))
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(LARGE[kind](rng), rng, 90), rng)
    _training_step(cell, p, forest, binding.PERSISTENT)


@pytest.mark.parametrize("kind", ["two callers", "itself", "cycle", "same children"])
def test_large_malformed_forests_return_errors(kind):
    """the ways are chosen from the arrays before anything has validated them"""
    rng = np.random.default_rng(950)
    p = fg.draw_recursive_params(rng, 20, 90, tensor=False, emb_scale=0.8, w_scale=0.2)
    forest = fg.forest_from_shapes([fg.balanced_shape(256)] * 2 + [None] * 200 if kind == "same children" else [fg.balanced_shape(1024)] * 2, rng, 90)
    left, right = forest.left.copy(), forest.right.copy()
    inner = np.flatnonzero(left >= 0)
    if kind == "two callers":
        left[inner[7]] = left[inner[300]]
    elif kind == "itself":
        right[inner[40]] = inner[40]
    elif kind == "cycle":                       # a node below the root calls the root
        left[inner[3]] = forest.roots[0]
    else:                                       # 202 trees by the node count, six times as many nodes without a caller
        left[inner], right[inner] = left[inner[0]], right[inner[0]]
    model = _model(binding.CELL_TREERNN, p)
    with pytest.raises(binding.TreeLSTMError) as err:
        model.forward(util.to_dev(left), util.to_dev(right), util.to_dev(forest.token), flags=binding.PERSISTENT)
    assert err.value.code == binding.ERR_INVALID_FOREST
    _check(binding.CELL_TREERNN, p, forest, binding.PERSISTENT)
    model.close()


@pytest.mark.parametrize("cell,n_trees,hi", [(binding.CELL_TREERNN, 20, 40), (binding.CELL_TREERNN, 1, 1),
                                             (binding.CELL_RNTN, 20, 24), (binding.CELL_RNTN, 1, 1)])
def test_label_out_of_range_reaches_no_gradient(cell, n_trees, hi):
    """a bad label ends the step before anything is added to a gradient (which tokens had got their row of
    dEmb_rows by then is a matter of timing): the cleared outputs stay zero, the memory behind the rows of the
    leaves is not touched, and the context takes the next step"""
    rng = np.random.default_rng(800 + hi)
    tensor = cell == binding.CELL_RNTN
    p = fg.draw_recursive_params(rng, 24, 50, tensor=tensor, emb_scale=0.8, w_scale=0.2, v_scale=0.02)
    forest = fg.random_forest(rng, n_trees, 1, hi, 50)
    n, leaves, H, C = forest.n_nodes, forest.n_leaves, p.H, 5
    model = _model(cell, p)
    model.set_classifier(util.to_dev(rng.uniform(-0.3, 0.3, size=(H, C)).astype(np.float32)), util.to_dev(np.zeros(C, np.float32)))
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
    labels = np.zeros(n, np.int32)
    labels[n // 2] = C
    model.forward(*arrs, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    f32 = dict(dtype=torch.float32, device="cuda")
    out = {k: torch.full(shape, 7.0, **f32) for k, shape in dict(loss=(1,), dW=(2 * H, H), db=(H,), dV=(H, 2 * H, 2 * H), dWc=(H, C), dbc=(C,)).items()}
    rows = torch.full((leaves + 8, H), 7.0, **f32)
    ids, touched = torch.empty(leaves, dtype=torch.int32, device="cuda"), torch.empty(1, dtype=torch.int32, device="cuda")
    bad = util.to_dev(labels)
    ptr = lambda t: t.data_ptr()
    rc_ = model.lib.treelstm_backward_recursive(model.handle, ptr(bad), ptr(out["loss"]), ptr(out["dW"]), ptr(out["db"]), ptr(out["dV"]),
                                                ptr(out["dWc"]), ptr(out["dbc"]), ptr(ids), ptr(rows), ptr(touched), None)
    assert rc_ == binding.OK and model.status_sync() == binding.ERR_LABEL_OUT_OF_RANGE
    assert bool((rows[leaves:] == 7.0).all()) and not bool(rows[:leaves].any())
    assert not bool(out["dW"].any()) and not bool(out["db"].any()) and (not tensor or not bool(out["dV"].any()))
    labels[n // 2] = 0
    model.forward(*arrs, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    assert np.isfinite(model.backward_recursive(util.to_dev(labels), leaves)["loss"].item())
    model.close()


@pytest.mark.parametrize("overlap", [0, 1])
@pytest.mark.parametrize("kind", ["sentences", "one large tree"])
def test_a_backward_pass_may_be_repeated(kind, overlap):
    """two backward passes behind one forward, on tree clusters and over the whole GPU"""
    rng = np.random.default_rng(960)
    p = fg.draw_recursive_params(rng, 20, 90, tensor=False, emb_scale=0.8, w_scale=0.2)
    shapes = [fg.random_split_shape(rng, 20) for _ in range(8)] if kind == "sentences" else [fg.balanced_shape(1024)] * 2
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 90), rng)
    Wc, bc = rng.uniform(-0.3, 0.3, size=(20, 3)).astype(np.float32), rng.uniform(-0.1, 0.1, size=3).astype(np.float32)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = rc.loss_and_gradients(KIND[binding.CELL_TREERNN], forest.left, forest.right, forest.token, p.emb, p.W, p.b, Wc, bc, labels, p.V)
    model = _model(binding.CELL_TREERNN, p)
    model.set_option(binding.OPT_OVERLAP_LAUNCH, overlap)
    model.set_classifier(util.to_dev(Wc), util.to_dev(bc))
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token, labels)]
    model.forward(*arrs[:3], flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    for _ in range(2):
        g = {k: v.cpu().numpy() for k, v in model.backward_recursive(arrs[3], forest.n_leaves).items()}
        util.compare_training_step(g, ref, util.TOL["fp32"], util.REL["fp32"], loss_rel=1e-5)
    model.close()


@pytest.mark.parametrize("cell,H", [(binding.CELL_TREERNN, 128), (binding.CELL_TREERNN, 20), (binding.CELL_RNTN, 32)])
@pytest.mark.parametrize("kind", ["one leaf", "few trees", "more trees than clusters", "left to the whole GPU"])
def test_states_are_the_same_with_and_without_a_backward_to_come(kind, cell, H):
    """two instantiations of the tree kernel: trees dealt by id, or by size with the lists kept; whose cluster a tree is changes no
    bit of its nodes' states (where both leave the forest to the whole GPU: neither)"""
    rng = np.random.default_rng(970 + H)
    p = fg.draw_recursive_params(rng, H, 90, tensor=cell == binding.CELL_RNTN, emb_scale=0.8, w_scale=1.0 / np.sqrt(2 * H), v_scale=1.0 / (2 * H))
    shapes = {"one leaf": [None], "few trees": [fg.random_split_shape(rng, int(n)) for n in rng.integers(2, 30, size=9)],
              "more trees than clusters": [None if t % 9 == 4 else fg.random_split_shape(rng, int(rng.integers(2, 6))) for t in range(160)],
              "left to the whole GPU": [fg.balanced_shape(1024 if H > 32 else 256)] * 2}[kind]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 90), rng)
    model = _model(cell, p)
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
    alone = model.forward(*arrs, flags=binding.PERSISTENT)["h"].cpu().numpy()
    saved = model.forward(*arrs, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)["h"].cpu().numpy()
    np.testing.assert_array_equal(alone, saved)
    model.close()
