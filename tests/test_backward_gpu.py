"""Parity of the CUDA training step (forward + backward through structure, via the C ABI) against
the fp64 oracle: loss and every gradient group within 1e-4 max-abs and within 2e-5 of the group's
own largest entry (several groups of the full-size workload lie below 1e-4 altogether)."""
import ctypes

import numpy as np
import pytest
import torch

from oracle import treelstm_oracle as orc
from paper_1809_00832_b200 import binding, forests as fg, trace
from tests import util

pytestmark = pytest.mark.gpu


def _train_step(model, forest, labels, flags):
    out = model.forward(util.to_dev(forest.left), util.to_dev(forest.right), util.to_dev(forest.token),
                        flags=flags | binding.SAVE_FOR_BACKWARD)
    grads = model.backward(util.to_dev(labels), forest.n_leaves)
    torch.cuda.synchronize()
    res = {k: v.cpu().numpy() for k, v in grads.items()}
    res["h"] = out["h"].cpu().numpy()
    return res


def _compare(res, ref, tol):
    util.compare_training_step(res, ref, tol, util.REL["fp32"], loss_rel=1e-5)


@pytest.mark.parametrize("flags", [binding.PER_LEVEL, binding.PERSISTENT])
def test_training_step_matches_oracle(flags):
    w = fg.make_workload("train25_fp32", 0)
    f, p = w.forest, w.params
    ref = orc.loss_and_gradients(f.left, f.right, f.token, p.emb, p.W, p.b, p.Wc, p.bc, w.labels)
    model = util.make_model(p, "fp32")
    res = _train_step(model, f, w.labels, flags)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    _compare(res, ref, util.TOL["fp32"])
    # gradients are overwritten, not accumulated: a second step gives the same numbers
    res2 = _train_step(model, f, w.labels, flags)
    _compare(res2, ref, util.TOL["fp32"])


@pytest.mark.parametrize("flags", [binding.PER_LEVEL, binding.PERSISTENT])
def test_training_step_full_size_with_large_gradients(flags):
    """the sizes of the training workload (H=150, E=300: 64 x 64 dW tiles, dIn chunks split over
    CTAs) with weights six times larger, so that every gradient group is far above the tolerance"""
    rng = np.random.default_rng(150)
    params = fg.draw_params(rng, 150, 300, 2000, emb_dist="normal", emb_scale=0.1, w_scale=0.3, n_classes=5)
    forest = fg.random_forest(rng, 25, 2, 56, 2000)
    forest, _ = fg.permute_node_ids(forest, rng)
    labels = rng.integers(0, 5, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b,
                                 params.Wc, params.bc, labels)
    for k in util.GRAD_KEYS + ("dEmb_rows",):
        assert np.max(np.abs(ref[k])) > 5 * util.TOL["fp32"], k      # the case has signal in every group
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, flags)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    _compare(res, ref, util.TOL["fp32"])


def test_training_step_small_odd_sizes_and_duplicates():
    # larger gradients (weights +-0.5), sizes that match no tile, permuted ids, duplicated tokens and
    # duplicated subtrees: every node must receive its own forward values
    rng = np.random.default_rng(4)
    params = fg.draw_params(rng, 7, 5, 6, emb_dist="uniform", emb_scale=0.5, w_scale=0.5, n_classes=3)
    shape = fg.random_split_shape(rng, 9)
    forest = fg.forest_from_shapes([shape, shape, None, fg.left_chain_shape(12)], rng, 6)
    forest, _ = fg.permute_node_ids(forest, rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b,
                                 params.Wc, params.bc, labels)
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    _compare(res, ref, util.TOL["fp32"])


def test_backward_errors():
    rng = np.random.default_rng(6)
    params = fg.draw_params(rng, 4, 4, 5, emb_dist="uniform", emb_scale=0.5, w_scale=0.5, n_classes=3)
    model = util.make_model(params, "fp32")
    forest = fg.forest_from_shapes([fg.random_split_shape(rng, 5)], rng, 5)
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
    labels = torch.zeros(forest.n_nodes, dtype=torch.int32, device="cuda")
    model.forward(*arrs, flags=binding.PERSISTENT)                  # nothing saved
    with pytest.raises(binding.TreeLSTMError) as err:
        model.backward(labels, forest.n_leaves)
    assert err.value.code == binding.ERR_STATE
    model.forward(*arrs, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    labels[2] = 3
    with pytest.raises(binding.TreeLSTMError) as err:
        model.backward(labels, forest.n_leaves)
    assert err.value.code == binding.ERR_LABEL_OUT_OF_RANGE


def test_data_parallel_step_single_rank():
    """the data-parallel wrapper on one rank: same gradients, touched rows trimmed to their count"""
    from paper_1809_00832_b200 import data_parallel
    w = fg.make_workload("train25_fp32", 0, n_trees=6)
    f, p = w.forest, w.params
    ref = orc.loss_and_gradients(f.left, f.right, f.token, p.emb, p.W, p.b, p.Wc, p.bc, w.labels)
    model = util.make_model(p, "fp32")
    out = data_parallel.training_step(model, util.to_dev(f.left), util.to_dev(f.right), util.to_dev(f.token),
                                      util.to_dev(w.labels), f.n_leaves, binding.PERSISTENT)
    res = {k: v.cpu().numpy() for k, v in out.items()}
    assert res["touched_ids"].shape[0] == len(ref["touched_ids"])
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("tensor_cores", [1, 0])
def test_weight_gradient_on_tensor_cores_and_on_fp32_units(tensor_cores):
    """dW and db of the one-launch backward, formed either by the split-bf16 tensor-core contraction
    (three bf16 pieces per fp32 value, six products per term) or by fp32 multiply-adds: both must meet
    the fp32 bounds against the oracle, on the full-size case with large gradients (several row tiles,
    a ragged last gate-column tile, several node runs) and on sizes that fill no tile"""
    rng = np.random.default_rng(151)
    cases = [(150, 300, 2000, fg.random_forest(rng, 25, 2, 56, 2000), 5, 0.3),
             (7, 5, 6, fg.forest_from_shapes([fg.random_split_shape(rng, 9), None, fg.left_chain_shape(70)], rng, 6), 3, 0.5)]
    for H, E, vocab, forest, n_classes, w_scale in cases:
        params = fg.draw_params(rng, H, E, vocab, emb_dist="normal", emb_scale=0.1, w_scale=w_scale, n_classes=n_classes)
        forest, _ = fg.permute_node_ids(forest, rng)
        labels = rng.integers(0, n_classes, size=forest.n_nodes).astype(np.int32)
        ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b,
                                     params.Wc, params.bc, labels)
        model = util.make_model(params, "fp32")
        model.set_option(binding.OPT_DW_TENSOR_CORES, tensor_cores)
        res = _train_step(model, forest, labels, binding.PERSISTENT)
        _compare(res, ref, util.TOL["fp32"])


def test_training_step_on_forests_of_single_leaves_and_with_a_large_vocabulary():
    """no internal node at all (the weight gradient's second part is empty, W_h gets zeros), and a
    vocabulary beyond what the token scan keeps in shared memory (its ballots are then read again)"""
    rng = np.random.default_rng(152)
    vocab = 400_000
    params = fg.draw_params(rng, 6, 4, vocab, emb_dist="uniform", emb_scale=0.5, w_scale=0.5, n_classes=3)
    for shapes in ([None, None, None], [fg.random_split_shape(rng, 40), None, fg.left_chain_shape(5)]):
        forest = fg.forest_from_shapes(shapes, rng, vocab)
        forest.token[int(np.flatnonzero(forest.left < 0)[0])] = vocab - 1   # the last id of the table is in use
        labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
        ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b,
                                     params.Wc, params.bc, labels)
        model = util.make_model(params, "fp32")
        for flags in (binding.PERSISTENT, binding.PER_LEVEL):
            res = _train_step(model, forest, labels, flags)
            _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("ctas", [1, 3, 40])
def test_training_step_on_small_grids(ctas):
    """the one-launch backward on a grid of one CTA (token scan and classifier in the same CTA), of a few
    CTAs (every CTA takes several blocks of a narrow wavefront, only the first of them fetched ahead of
    the grid barrier) and of fewer CTAs than a narrow wavefront has blocks"""
    rng = np.random.default_rng(160 + ctas)
    params = fg.draw_params(rng, 20, 12, 300, emb_dist="normal", emb_scale=0.3, w_scale=0.3, n_classes=4)
    forest = fg.random_forest(rng, 9, 2, 40, 300)
    forest, _ = fg.permute_node_ids(forest, rng)
    labels = rng.integers(0, 4, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b,
                                 params.Wc, params.bc, labels)
    model = util.make_model(params, "fp32")
    model.set_option(binding.OPT_MAX_CTAS, ctas)
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,E,n_trees,hi", [(25, 9, 40, 30), (103, 40, 20, 30), (161, 30, 12, 24), (256, 70, 8, 20), (257, 20, 3, 12), (150, 520, 2, 600)])
def test_training_step_at_the_limits_of_the_tree_kernels(H, E, n_trees, hi):
    """hidden sizes at which the cluster grows and at which the tree kernels end; more trees than clusters; states
    that do not fit the shared memory of a cluster; long embedding rows"""
    rng = np.random.default_rng(800 + H)
    params = fg.draw_params(rng, H, E, 90, emb_dist="normal", emb_scale=0.3, w_scale=1.0 / np.sqrt(H), n_classes=3)
    forest = fg.concat_forests([fg.random_forest(rng, n_trees, 1 if hi < 100 else hi - 1, hi, 90),
                                fg.forest_from_shapes([fg.left_chain_shape(9), fg.balanced_shape(32)], rng, 90)])
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,E,shapes", [
    (40, 30, "balanced"), (72, 127, "bushy"), (150, 64, "bushy"), (33, 128, "leaves"), (128, 63, "exact"), (256, 300, "bushy"), (300, 20, "balanced")])
def test_training_step_of_wide_forests(H, E, shapes):
    """forests whose wavefronts go over the whole GPU, their contractions on split bf16 pieces: wavefronts around 64,
    128 and 256 positions that start inside a block, ragged outputs and gate columns, the boundary between leaves and
    internal nodes inside a block or on it, narrow wavefronts on top, single leaves, sizes beyond the tree kernels"""
    rng = np.random.default_rng(900 + H)
    vocab = 70
    params = fg.draw_params(rng, H, E, vocab, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    if shapes == "balanced":
        forest = fg.forest_from_shapes([fg.balanced_shape(512)] * 2 + [None] * 3, rng, vocab)
    elif shapes == "exact":
        forest = fg.forest_from_shapes([fg.balanced_shape(1024)], rng, vocab)
    elif shapes == "leaves":
        forest = fg.forest_from_shapes([fg.balanced_shape(256)] * 2 + [None] * 600 + [fg.left_chain_shape(150)], rng, vocab)
    else:
        forest = fg.forest_from_shapes([fg.random_split_shape(rng, 701), fg.random_split_shape(rng, 390)], rng, vocab)
    forest, _ = fg.permute_node_ids(forest, rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    _compare(res, ref, util.TOL["fp32"])
    _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,trees", [(260, 256), (260, 257), (258, 257), (264, 128), (257, 129)])
def test_wide_wavefronts_at_the_limits_of_their_kinds(H, trees):
    """wavefronts of 256 and 257 nodes (operands formed at the tensor core or stored first), of exactly one and of one more
    than one tile of 128, in rows that can be read 16 bytes at a time and in rows that cannot"""
    rng = np.random.default_rng(77 + H + trees)
    params = fg.draw_params(rng, H, 20, 50, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    forest = fg.forest_from_shapes([fg.balanced_shape(4)] * trees, rng, 50)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,classes", [(40, 1), (64, 8), (64, 9), (65, 5), (65, 6), (160, 5), (161, 5), (256, 5), (256, 6), (257, 5)])
def test_classifier_of_every_width(H, classes):
    """the classifier's sums in registers up to 64, 160 and 256 units with few classes, in shared memory beyond"""
    rng = np.random.default_rng(H + classes)
    params = fg.draw_params(rng, H, 24, 40, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=classes)
    forest = fg.forest_from_shapes([fg.random_split_shape(rng, 30) for _ in range(4)] + [None], rng, 40)
    labels = rng.integers(0, classes, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,shapes", [(40, "one large tree"), (40, "chains"), (33, "leaves"), (150, "chains"), (200, "sentences")])
def test_large_forests_on_either_way(H, shapes):
    """forests beyond those that always go to the clusters, decided from the fullest cluster and the depth: one large tree
    among small ones and wide wavefronts go over the whole GPU, few deep trees and many small ones to the clusters"""
    rng = np.random.default_rng(1000 + H)
    params = fg.draw_params(rng, H, 30, 70, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    shape = {"one large tree": lambda: [fg.balanced_shape(512)] + [fg.random_split_shape(rng, 12) for _ in range(20)],
             "chains": lambda: [fg.left_chain_shape(150), fg.left_chain_shape(70)] + [fg.random_split_shape(rng, 20)],
             "leaves": lambda: [fg.balanced_shape(256)] * 2 + [None] * 600,
             "sentences": lambda: [fg.random_split_shape(rng, int(n)) for n in rng.integers(1, 40, size=30)]}[shapes]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shape(), rng, 70), rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,n_trees", [(150, 15), (150, 16), (150, 61), (20, 147), (20, 148), (20, 512), (20, 513)])
def test_trees_dealt_by_size(H, n_trees):
    """as many trees as clusters (15 and 147 on 148 SMs), one more, as many as are dealt by size at most, one more; sizes far
    apart, trees of one leaf among them, and one cluster whose lists are longer than what the forward keeps for the backward"""
    rng = np.random.default_rng(1200 + H + n_trees)
    params = fg.draw_params(rng, H, 24, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    shapes = [fg.left_chain_shape(90), fg.random_split_shape(rng, 50)] + [
        None if t % 11 == 3 else fg.random_split_shape(rng, int(rng.integers(2, 4 if n_trees > 100 else 24))) for t in range(n_trees - 2)]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 60), rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("vocab,trees,ctas", [
    (1, (3, 2), 0), (2, (5, 1), 0), (127, (40, 5), 0), (128, (40, 5), 0), (129, (40, 5), 0), (37888, (60, 9), 0), (37889, (60, 9), 0),
    (65536, (60, 9), 2), (65537, (60, 9), 2), (300, (6000, 2000), 0), (300, (6001, 1998), 0)])
def test_touched_tokens_and_their_rows(vocab, trees, ctas):
    """one id, groups of 128 ids with a partial one, one and two groups a CTA on 148 SMs, as many ids as two CTAs keep and one more; the
    largest forest whose tokens are found by the CTAs that number them (20000 nodes) and one of 20001.  First and last id are in use"""
    rng = np.random.default_rng(vocab + trees[0])
    H, E = 8, 8
    params = fg.draw_params(rng, H, E, vocab, emb_dist="normal", emb_scale=0.3, w_scale=0.25, n_classes=3)
    shapes = [fg.balanced_shape(2)] * trees[0] + [None] * trees[1]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, vocab), rng)
    leaves = np.flatnonzero(forest.left < 0)
    forest.token[leaves[0]], forest.token[leaves[-1]] = 0, vocab - 1
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    if ctas:
        model.set_option(binding.OPT_MAX_CTAS, ctas)
    res = _train_step(model, forest, labels, binding.PERSISTENT)
    m = int(res["n_touched"][0])
    assert m == len(ref["touched_ids"])
    assert np.array_equal(res["touched_ids"][:m], ref["touched_ids"])
    _compare(res, ref, util.TOL["fp32"])


@pytest.mark.parametrize("precision,n_trees", [("fp32", 6), ("bf16", 6), ("fp32", 90), ("bf16", 90)])
def test_weights_of_the_backward_come_with_the_classifier_and_follow_every_update(precision, n_trees):
    """a context without a classifier keeps no weights in the layouts that only the backward reads; the classifier may come
    between forward and backward; new weights reach every layout (tree clusters and wide wavefronts)"""
    rng = np.random.default_rng(1100 + n_trees)
    draw = lambda: fg.draw_params(rng, 256, 300, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.04, n_classes=3)
    params, other = draw(), draw()
    forest = fg.random_forest(rng, n_trees, 2, 30, 60)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    util.lib_ready()
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token, labels)]
    weights = [[util.to_dev(a) for a in (p.emb, p.W, p.b, p.Wc, p.bc)] for p in (params, other)]
    create = lambda: binding.TreeLSTM(256, 300, 60, *weights[0][:3], binding.FP32 if precision == "fp32" else binding.BF16)
    create().close()                                              # the kernels that a create launches are on the device now
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    model = create()
    assert before - torch.cuda.mem_get_info()[0] <= 12 << 20      # W 4.2 MB and one image of it; with the backward's two: 16 and more
    need = model.workspace_bytes(forest.n_nodes, True)
    model.forward(*arrs[:3], flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    model.set_classifier(*weights[0][3:])
    assert model.workspace_bytes(forest.n_nodes, True) == need
    for k, p in ((0, params), (1, other)):
        if k:
            model.update_weights(*weights[1][:3])
            model.set_classifier(*weights[1][3:])
            model.forward(*arrs[:3], flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
        res = {q: v.cpu().numpy() for q, v in model.backward(arrs[3], forest.n_leaves).items()}
        ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, p.emb, p.W, p.b, p.Wc, p.bc, labels)
        for q in ("dW", "db", "dWc", "dbc"):
            assert util.max_abs(res[q], ref[q]) <= util.REL[precision] * float(np.abs(ref[q]).max()), q
        n = int(res["n_touched"][0])
        assert util.max_abs(res["dEmb_rows"][:n], ref["dEmb_rows"]) <= util.REL[precision] * float(np.abs(ref["dEmb_rows"]).max())
    model.close()


class _RawStep:
    """forward that keeps its activations and backward as a C caller enqueues them, with a workspace of their own, on the current
    stream; nothing waits for the device"""

    def __init__(self, model, forest, labels):
        f32, i32 = dict(dtype=torch.float32, device="cuda"), dict(dtype=torch.int32, device="cuda")
        n, H, E, C = forest.n_nodes, model.H, model.E, model.C
        self.model, self.n = model, n
        self.forest = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
        self.labels = util.to_dev(labels)
        self.states = [torch.empty((n, H), **f32), torch.empty((n, H), **f32), torch.empty(n, **i32), torch.empty(n, **i32),
                       torch.empty(n + 2, **i32), torch.empty(1, **i32)]
        self.grads = dict(loss=torch.empty(1, **f32), dW=torch.empty((E + 2 * H, 5 * H), **f32), db=torch.empty(5 * H, **f32),
                          dWc=torch.empty((H, C), **f32), dbc=torch.empty(C, **f32), touched_ids=torch.empty(forest.n_leaves, **i32),
                          dEmb_rows=torch.empty((forest.n_leaves, E), **f32), n_touched=torch.empty(1, **i32))
        need = model.workspace_bytes(n, True)
        self.ws = torch.empty(need + 256, dtype=torch.uint8, device="cuda")
        self.at, self.ws_bytes = self.ws.data_ptr() + (-self.ws.data_ptr()) % 256, need

    def forward(self):
        rc = self.model.lib.treelstm_forward(self.model.handle, self.n, *(t.data_ptr() for t in self.forest + self.states),
                                             binding.PERSISTENT | binding.SAVE_FOR_BACKWARD, self.at, self.ws_bytes,
                                             torch.cuda.current_stream().cuda_stream)
        assert rc == binding.OK

    def backward(self):
        rc = self.model.lib.treelstm_backward(self.model.handle, self.labels.data_ptr(), *(t.data_ptr() for t in self.grads.values()),
                                              torch.cuda.current_stream().cuda_stream)
        assert rc == binding.OK


@pytest.mark.parametrize("call", ["forward_host", "per_level"])
def test_backward_that_ends_beside_another_call_leaves_its_answer_alone(call):
    """a backward pass (one whose labels are bad) is left on its stream while a call on another stream waits for its own level and
    root counts and status; the backward ends before, within and behind that call"""
    rng = np.random.default_rng(1400)
    params = fg.draw_params(rng, 20, 12, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.3, n_classes=3)
    model = util.make_model(params, "fp32")
    model.set_option(binding.OPT_MAX_CTAS, 16)                   # the kernels of both streams fit the device together
    one = fg.forest_from_shapes([fg.left_chain_shape(30), None], rng, 60)
    other = fg.forest_from_shapes([fg.balanced_shape(4)] * 5, rng, 60)
    labels = rng.integers(0, 3, size=one.n_nodes).astype(np.int32)
    labels[3] = 3
    step = _RawStep(model, one, labels)
    host = binding.pack_forest_host(other.left, other.right, other.token)
    dev = [util.to_dev(a) for a in (other.left, other.right, other.token)]
    want = {k: v.cpu().numpy() for k, v in model.forward(*dev, flags=binding.PER_LEVEL).items()}
    roots = model.forward_host(*host, max_roots=8)["root_h"].numpy().copy()
    out, levels = model.forward_host(*host, max_roots=8), model.forward(*dev, flags=binding.PER_LEVEL)
    behind, beside = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for wait in range(0, 400):
        with torch.cuda.stream(behind):
            step.forward()
            torch.cuda._sleep(500 * wait)                        # cycles: up to 100 us
            step.backward()
        with torch.cuda.stream(beside):
            if call == "forward_host":
                model.forward_host(*host, max_roots=8, out=out)
                assert int(out["n_levels"]) == 3 and int(out["n_roots"]) == 5
                np.testing.assert_array_equal(out["root_h"].numpy()[:5], roots[:5])
            else:
                model.forward(*dev, flags=binding.PER_LEVEL, out=levels)   # one launch a level, as many as the host has read
                np.testing.assert_array_equal(levels["h"].cpu().numpy(), want["h"])
        behind.synchronize()


def test_status_of_the_last_backward_when_one_on_another_stream_ends_later():
    """two backward passes on two streams with a workspace each: treelstm_status_sync speaks of the last call, whichever of them
    is the last to end"""
    rng = np.random.default_rng(1401)
    params = fg.draw_params(rng, 20, 12, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.3, n_classes=3)
    model = util.make_model(params, "fp32")
    model.set_option(binding.OPT_MAX_CTAS, 16)
    forest = fg.forest_from_shapes([fg.left_chain_shape(30), fg.balanced_shape(4)], rng, 60)
    good = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    bad = good.copy()
    bad[5] = 3
    steps = {binding.OK: _RawStep(model, forest, good), binding.ERR_LABEL_OUT_OF_RANGE: _RawStep(model, forest, bad)}
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    for last, first in ((binding.OK, binding.ERR_LABEL_OUT_OF_RANGE), (binding.ERR_LABEL_OUT_OF_RANGE, binding.OK)):
        for first_ends_later in (False, True):
            torch.cuda.synchronize()
            with torch.cuda.stream(streams[0]):
                steps[first].forward()
                torch.cuda._sleep(20_000_000 if first_ends_later else 1)      # 10 ms
                steps[first].backward()
            if not first_ends_later:
                streams[0].synchronize()
            with torch.cuda.stream(streams[1]):
                steps[last].forward()
                steps[last].backward()
            assert model.status_sync() == last
            torch.cuda.synchronize()
            assert model.status_sync() == last                   # the other one's word lies there now
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, good)
    _compare({k: v.cpu().numpy() for k, v in steps[binding.OK].grads.items()}, ref, util.TOL["fp32"])


REPEATED = {
    "tree clusters": (150, lambda rng: [fg.random_split_shape(rng, int(n)) for n in rng.integers(2, 40, size=20)]),
    "wide wavefronts": (40, lambda rng: [fg.balanced_shape(512)] * 2 + [None] * 3),
    "beyond the tree kernels": (300, lambda rng: [fg.balanced_shape(64)] * 2),
}


@pytest.mark.parametrize("overlap", [0, 1])
@pytest.mark.parametrize("kind", REPEATED)
def test_a_backward_pass_may_be_repeated(kind, overlap):
    """two backward passes behind one forward, on every way through the forest and with either launch form of the forward: the second
    finds the counters of its grid barriers as the first one did"""
    H, shapes = REPEATED[kind]
    rng = np.random.default_rng(1500 + H)
    params = fg.draw_params(rng, H, 30, 70, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes(rng), rng, 70), rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    model.set_option(binding.OPT_OVERLAP_LAUNCH, overlap)
    arrs = [util.to_dev(a) for a in (forest.left, forest.right, forest.token, labels)]
    model.forward(*arrs[:3], flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    for _ in range(2):
        _compare({k: v.cpu().numpy() for k, v in model.backward(arrs[3], forest.n_leaves).items()}, ref, util.TOL["fp32"])


def test_backward_passes_side_by_side_share_the_device():
    """two contexts' backward passes of wide forests, each with a grid barrier over the whole device, enqueued on two streams at once"""
    rng = np.random.default_rng(1600)
    params = fg.draw_params(rng, 40, 30, 70, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(40), n_classes=3)
    forest = fg.forest_from_shapes([fg.balanced_shape(512)] * 4, rng, 70)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    models = [util.make_model(params, "fp32") for _ in range(2)]
    steps = [_RawStep(m, forest, labels) for m in models]
    streams = [torch.cuda.Stream() for _ in models]
    torch.cuda.synchronize()
    for _ in range(10):
        for step in steps:                                        # (one after the other: a forward has the device to itself)
            step.forward()
            torch.cuda.synchronize()
        for step, stream in zip(steps, streams):
            with torch.cuda.stream(stream):
                torch.cuda._sleep(100_000)                        # both are enqueued by the time either starts
                step.backward()
        assert [m.status_sync() for m in models] == [binding.OK] * 2
    for step in steps:
        _compare({k: v.cpu().numpy() for k, v in step.grads.items()}, ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,trees", [(300, 40), (300, 150), (520, 40), (520, 700)])
def test_rows_that_the_kernel_ahead_numbers(H, trees):
    """hidden sizes without tree kernels, where the launch ahead of the weight gradient numbers the embedding gradient's rows: forests of single leaves,
    whose pass ends with that numbering; other words from step to step in the same memory, so that rows of the step before are never the right ones"""
    rng = np.random.default_rng(H + trees)
    vocab, E = 3000, 20
    params = fg.draw_params(rng, H, E, vocab, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    model = util.make_model(params, "fp32")
    for step in range(4):
        forest = fg.forest_from_shapes([None] * trees, rng, vocab)
        words = rng.choice(vocab, size=5 + 40 * step, replace=False).astype(np.int32)       # each of them several times, in any order
        forest.token[:] = words[rng.integers(0, len(words), size=trees)]
        labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
        ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                     params.bc, labels)
        _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])


@pytest.mark.parametrize("H,kind,kept", [(150, "planned", True), (150, "one tree", True), (20, "one tree", True), (20, "more nodes than are planned ahead", True),
                                         (20, "more depths than are planned ahead", False)])
def test_lists_of_the_forward_are_kept_for_the_backward(H, kind, kept):
    """planned beside the leaves, behind the clusters' own blocks where one cluster has all of them, and by the clusters themselves where the planning CTA has no
    room: the backward plans nothing itself (trace build: that would leave a stamp), unless lists that clusters have planned are longer than their blocks"""
    rng = np.random.default_rng(301)
    params = fg.draw_params(rng, H, 12, 40, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    shapes = {"planned": [fg.random_split_shape(rng, int(k)) for k in range(2, 40)], "one tree": [fg.left_chain_shape(300)],
              "more nodes than are planned ahead": [fg.left_chain_shape(29)] * 300,
              "more depths than are planned ahead": [fg.left_chain_shape(400)] + [fg.left_chain_shape(2)] * 200}[kind]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 40), rng)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32", variant="trace")
    model._workspace(forest.n_nodes, True).zero_()
    _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])
    setup = trace.read_trace(model, 1)[trace.LEVELS - 1]
    assert setup[3] > 0 and (setup[6] == 0) == kept                       # (dealt; depth 255 of a chain shares this row's first six slots)


@pytest.mark.parametrize("H,chains", [(64, 128), (96, 129), (150, 128), (224, 128), (224, 129), (256, 129)])
def test_wavefronts_of_one_and_two_tiles(H, chains):
    """wavefronts of 128, 129 to 192, 256 and 257 nodes in a forest that the tree kernels leave: operands formed at the tensor core (one tile; two, where the
    rows are whole lines and no CTA forms two blocks) or stored first"""
    rng = np.random.default_rng(400 + H + chains)
    params = fg.draw_params(rng, H, 20, 50, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    forest = fg.forest_from_shapes([fg.left_chain_shape(12)] * chains + [fg.balanced_shape(1024)], rng, 50)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    _compare(_train_step(model, forest, labels, binding.PERSISTENT), ref, util.TOL["fp32"])


@pytest.mark.parametrize("words", [1, 2, 3])
@pytest.mark.parametrize("H,E,shapes", [(40, 24, "sentences"), (42, 26, "sentences"), (33, 23, "sentences"), (40, 24, "wide"), (300, 20, "sentences")])
def test_gradients_in_memory_of_any_alignment(H, E, shapes, words):
    """outputs that start 4, 8 and 12 bytes behind a 16-byte boundary (rows added in pieces of one, two and four floats, by the address and the
    width): behind the tree kernels, from the images of a wide forest, and where neither applies; what lies around them stays"""
    rng = np.random.default_rng(500 + H)
    params = fg.draw_params(rng, H, E, 70, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    forest = fg.forest_from_shapes([fg.balanced_shape(512)] * 2 if shapes == "wide" else [fg.random_split_shape(rng, k) for k in (20, 9, 1, 14)], rng, 70)
    labels = rng.integers(0, 3, size=forest.n_nodes).astype(np.int32)
    ref = orc.loss_and_gradients(forest.left, forest.right, forest.token, params.emb, params.W, params.b, params.Wc,
                                 params.bc, labels)
    model = util.make_model(params, "fp32")
    arrays = [util.to_dev(a) for a in (forest.left, forest.right, forest.token)]
    on_device = util.to_dev(labels)
    out = model.forward(*arrays, flags=binding.PERSISTENT | binding.SAVE_FOR_BACKWARD)
    shape = dict(dW=(E + 2 * H, 5 * H), db=(5 * H,), dWc=(H, 3), dbc=(3,), dEmb_rows=(forest.n_leaves, E))
    whole = {k: torch.full((int(np.prod(v)) + 8,), 7.0, device="cuda") for k, v in shape.items()}
    at = {k: v[words:words + int(np.prod(shape[k]))] for k, v in whole.items()}
    loss, touched, count = torch.empty(1, device="cuda"), *(torch.empty(k, dtype=torch.int32, device="cuda") for k in (forest.n_leaves, 1))
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())
    rc = model.lib.treelstm_backward(model.handle, ptr(on_device), ptr(loss), ptr(at["dW"]), ptr(at["db"]), ptr(at["dWc"]), ptr(at["dbc"]), ptr(touched),
                                     ptr(at["dEmb_rows"]), ptr(count), binding._stream())
    assert rc == binding.OK and model.status_sync() == binding.OK
    for k, v in whole.items():
        v = v.cpu().numpy()
        assert (v[:words] == 7.0).all() and (v[words + int(np.prod(shape[k])):] == 7.0).all(), k
    res = {k: v.cpu().numpy().reshape(shape[k]) for k, v in at.items()}
    res.update(loss=loss.cpu().numpy(), touched_ids=touched.cpu().numpy(), n_touched=count.cpu().numpy())
    _compare(res, ref, util.TOL["fp32"])
    del out
