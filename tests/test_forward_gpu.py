"""Parity of the CUDA forward path (through the C ABI) against the fp64 oracle on the same seeded
forests: schedule bit-exact, h and c within 1e-4 (fp32) / 3e-2 (bf16 operands)."""
import numpy as np
import pytest
import torch

from oracle import treelstm_oracle as orc
from paper_1809_00832_b200 import binding, forests as fg, trace
from tests import util

pytestmark = pytest.mark.gpu

MODES = [binding.PER_LEVEL, binding.PERSISTENT]


@pytest.mark.parametrize("flags", MODES)
@pytest.mark.parametrize("name", ["tiny8", "batch25_fp32"])
def test_fp32_forward_matches_oracle(name, flags):
    w = fg.make_workload(name, 0)
    ref = util.oracle_forward_cached(name, 0)
    model = util.make_model(w.params, "fp32")
    res = util.gpu_forward(model, w.forest, flags)
    util.check_schedule(res, ref, w.forest.n_nodes)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]
    assert util.max_abs(res["c"], ref["c"]) < util.TOL["fp32"]
    assert model.last_launch_count() >= 2


@pytest.mark.parametrize("single_cta", [True, False])
def test_schedule_paths_agree_with_oracle_on_permuted_ids(single_cta):
    rng = np.random.default_rng(11)
    w = fg.make_workload("batch25_fp32", 3)
    forest, new_of_old = fg.permute_node_ids(w.forest, rng)
    status, parent, level, order, off = orc.schedule(forest.left, forest.right)
    model = util.make_model(w.params, "fp32")
    if not single_cta:
        model.set_option(binding.OPT_SCHED_SINGLE_CTA_MAX, 0)
    res = util.gpu_forward(model, forest, binding.PERSISTENT)
    util.check_schedule(res, dict(level=level, order=order, level_offset=off), forest.n_nodes)
    # the recursive formulation does not depend on the numbering: same state per node
    href, cref, _ = orc.forward_recursive(forest.left, forest.right, forest.token, w.params.emb,
                                          w.params.W, w.params.b)
    assert util.max_abs(res["h"], href) < util.TOL["fp32"]
    assert util.max_abs(res["c"], cref) < util.TOL["fp32"]
    roots = model.roots(forest.n_trees + 3)
    torch.cuda.synchronize()
    n_roots = int(roots["n_roots"].item())
    assert n_roots == forest.n_trees
    ids = roots["root_ids"].cpu().numpy()[:n_roots]
    np.testing.assert_array_equal(ids, np.sort(forest.roots))
    np.testing.assert_array_equal(roots["root_h"].cpu().numpy()[:n_roots], res["h"][ids])
    np.testing.assert_array_equal(roots["root_c"].cpu().numpy()[:n_roots], res["c"][ids])
    res0 = util.gpu_forward(model, w.forest, binding.PERSISTENT)
    np.testing.assert_allclose(res["h"][new_of_old], res0["h"], atol=2e-6)


@pytest.mark.parametrize("single_cta", [True, False])
def test_deep_and_wide_schedules(single_cta):
    """closed-form shapes: chains (many levels, more than one radix digit) and balanced trees"""
    rng = np.random.default_rng(0)
    params = fg.draw_params(rng, 8, 8, 50, emb_dist="uniform", emb_scale=0.1, w_scale=0.1)
    model = util.make_model(params, "fp32")
    if not single_cta:
        model.set_option(binding.OPT_SCHED_SINGLE_CTA_MAX, 0)
    chain = fg.forest_from_shapes([fg.left_chain_shape(300), fg.left_chain_shape(5)], rng, 50)
    res = util.gpu_forward(model, chain, binding.PERSISTENT)
    status, _, level, order, off = orc.schedule(chain.left, chain.right)
    util.check_schedule(res, dict(level=level, order=order, level_offset=off), chain.n_nodes)
    assert res["n_levels"] == 300
    href, cref, _ = orc.forward_recursive(chain.left, chain.right, chain.token, params.emb, params.W, params.b)
    assert util.max_abs(res["h"], href) < util.TOL["fp32"]
    bal = fg.forest_from_shapes([fg.balanced_shape(256)] * 3, rng, 50)
    res = util.gpu_forward(model, bal, binding.PER_LEVEL)
    assert np.diff(res["level_offset"][:10]).tolist() == [3 * 256 >> k for k in range(9)]
    href, cref, _ = orc.forward_recursive(bal.left, bal.right, bal.token, params.emb, params.W, params.b)
    assert util.max_abs(res["h"], href) < util.TOL["fp32"]
    assert util.max_abs(res["c"], cref) < util.TOL["fp32"]


def test_large_forest_uses_multi_cta_schedule():
    """more nodes than the single-CTA scheduler takes (32768): properties that hold at any size plus
    sampled trees against the oracle"""
    rng = np.random.default_rng(5)
    params = fg.draw_params(rng, 16, 16, 100, emb_dist="uniform", emb_scale=0.1, w_scale=0.1)
    forest = fg.random_forest(rng, 2200, 2, 56, 100)
    assert forest.n_nodes > 32768
    model = util.make_model(params, "fp32")
    res = util.gpu_forward(model, forest, binding.PERSISTENT)
    status, _, level, order, off = orc.schedule(forest.left, forest.right)
    util.check_schedule(res, dict(level=level, order=order, level_offset=off), forest.n_nodes)
    sample = [0, 7, 1100, 2199]
    sub = fg.select_trees(forest, sample)
    href, cref, _ = orc.forward_recursive(sub.left, sub.right, sub.token, params.emb, params.W, params.b)
    ids = np.nonzero(np.isin(forest.tree_of, sample))[0]
    assert util.max_abs(res["h"][ids], href) < util.TOL["fp32"]
    assert util.max_abs(res["c"][ids], cref) < util.TOL["fp32"]


def test_edge_cases():
    rng = np.random.default_rng(1)
    params = fg.draw_params(rng, 5, 3, 9, emb_dist="uniform", emb_scale=0.5, w_scale=0.5)
    model = util.make_model(params, "fp32")
    # empty forest
    empty = fg.Forest(*(np.zeros(0, dtype=np.int32) for _ in range(5)))
    for flags in MODES:
        res = util.gpu_forward(model, empty, flags)
        assert res["n_levels"] == 0
    # single leaf, forest of leaves only, and H, E that are not multiples of any tile size
    for shapes in ([None], [None] * 70, [fg.random_split_shape(rng, 3), None]):
        forest = fg.forest_from_shapes(shapes, rng, 9)
        for flags in MODES:
            res = util.gpu_forward(model, forest, flags)
            href, cref, _ = orc.forward_recursive(forest.left, forest.right, forest.token, params.emb,
                                                  params.W, params.b)
            assert util.max_abs(res["h"], href) < util.TOL["fp32"]
            assert util.max_abs(res["c"], cref) < util.TOL["fp32"]


@pytest.mark.parametrize("single_cta", [True, False])
@pytest.mark.parametrize("flags", MODES)
def test_malformed_forests_return_errors(single_cta, flags):
    rng = np.random.default_rng(2)
    params = fg.draw_params(rng, 4, 4, 5, emb_dist="uniform", emb_scale=0.5, w_scale=0.5)
    model = util.make_model(params, "fp32")
    if not single_cta:
        model.set_option(binding.OPT_SCHED_SINGLE_CTA_MAX, 0)
    cases = [
        ([-1, -1, 0], [-1, -1, 3], [0, 1, -1], binding.ERR_INVALID_FOREST),       # child out of range
        ([-1, -1, 0], [-1, -1, -1], [0, 1, 2], binding.ERR_INVALID_FOREST),       # one child only
        ([-1, -1, 0, 0], [-1, -1, 1, 1], [0, 1, 0, 0], binding.ERR_INVALID_FOREST),  # two parents
        ([-1, -1, 0], [-1, -1, 0], [0, 1, 0], binding.ERR_INVALID_FOREST),        # same child twice
        ([-1, -1, 2], [-1, -1, 1], [0, 1, 0], binding.ERR_INVALID_FOREST),        # own child
        ([-1, 2, 1, -1], [-1, 0, 3, -1], [0, 0, 0, 0], binding.ERR_INVALID_FOREST),  # cycle
        ([-1, -1, 0], [-1, -1, 1], [5, 1, -1], binding.ERR_TOKEN_OUT_OF_RANGE),
        ([-1, -1, 0], [-1, -1, 1], [-2, 1, -1], binding.ERR_TOKEN_OUT_OF_RANGE),
    ]
    for l, r, t, code in cases:
        arrs = [torch.tensor(x, dtype=torch.int32, device="cuda") for x in (l, r, t)]
        assert orc.schedule(np.array(l, dtype=np.int32), np.array(r, dtype=np.int32), np.array(t, dtype=np.int32),
                            5)[0] == code
        with pytest.raises(binding.TreeLSTMError) as err:
            model.forward(*arrs, flags=flags)
        assert err.value.code == code
    # the context stays usable
    good = fg.forest_from_shapes([fg.random_split_shape(rng, 6)], rng, 5)
    res = util.gpu_forward(model, good, flags)
    href, _, _ = orc.forward_recursive(good.left, good.right, good.token, params.emb, params.W, params.b)
    assert util.max_abs(res["h"], href) < util.TOL["fp32"]


def test_argument_errors():
    rng = np.random.default_rng(3)
    params = fg.draw_params(rng, 4, 4, 5, emb_dist="uniform", emb_scale=0.5, w_scale=0.5)
    model = util.make_model(params, "fp32")
    lib = model.lib
    z = torch.zeros(8, dtype=torch.int32, device="cuda")
    f = torch.zeros(8, 4, device="cuda")
    ws = torch.zeros(1 << 16, dtype=torch.uint8, device="cuda")
    p = lambda t: None if t is None else __import__("ctypes").c_void_p(t.data_ptr())
    # workspace too small
    rc = lib.treelstm_forward(model.handle, 8, p(z), p(z), p(z), p(f), p(f), p(z), p(z), None, p(z), 0, p(ws), 16, None)
    assert rc == binding.ERR_INVALID_ARG
    rc = lib.treelstm_forward(model.handle, 8, None, p(z), p(z), p(f), p(f), p(z), p(z), None, p(z), 0, p(ws), 1 << 16, None)
    assert rc == binding.ERR_INVALID_ARG
    rc = lib.treelstm_forward(model.handle, 8, p(z), p(z), p(z), p(f), p(f), p(z), p(z), None, p(z), 64, p(ws), 1 << 16, None)
    assert rc == binding.ERR_INVALID_ARG
    assert lib.treelstm_backward(model.handle, p(z), p(f), p(f), p(f), p(f), p(f), p(z), p(f), p(z), None) == binding.ERR_STATE


def test_host_buffer_forward():
    w = fg.make_workload("tiny8", 0)
    ref = util.oracle_forward_cached("tiny8", 0)
    model = util.make_model(w.params, "fp32")
    f = w.forest
    host = [torch.from_numpy(a).pin_memory() for a in (f.left, f.right, f.token)]
    out = model.forward_host(*host, all_states=True, max_roots=f.n_trees)
    assert int(out["n_levels"][0]) == len(ref["level_offset"]) - 1
    assert int(out["n_roots"][0]) == f.n_trees
    np.testing.assert_array_equal(out["order"].numpy(), ref["order"])
    assert util.max_abs(out["h"].numpy(), ref["h"]) < util.TOL["fp32"]
    np.testing.assert_array_equal(out["root_ids"].numpy(), np.sort(f.roots))
    assert util.max_abs(out["root_h"].numpy(), ref["h"][np.sort(f.roots)]) < util.TOL["fp32"]
    assert util.max_abs(out["root_c"].numpy(), ref["c"][np.sort(f.roots)]) < util.TOL["fp32"]
    # roots only, second call reuses the library's staging buffers
    out2 = model.forward_host(*host, max_roots=f.n_trees)
    np.testing.assert_array_equal(out2["root_h"].numpy(), out["root_h"].numpy())


def test_roots_into_memory_that_is_pinned_in_part():
    """a registered range that ends before the last of max_roots rows: the kernel does not write there; the copy either
    takes such memory or says that it does not, and the next call is not troubled by it"""
    w = fg.make_workload("tiny8", 0)
    f, H, m = w.forest, w.params.H, w.forest.n_nodes            # room for as many roots as there are nodes
    model = util.make_model(w.params, "fp32")
    host = [torch.from_numpy(a).pin_memory() for a in (f.left, f.right, f.token)]
    good = model.forward_host(*host, max_roots=f.n_trees)
    page = 4096
    rows = (m * H * 4 + page - 1) // page + 1
    raw = np.full((2 * rows + 2) * page, 7, np.uint8)
    first = -raw.ctypes.data % page
    root_h = torch.from_numpy(raw[first:first + m * H * 4].view(np.float32)).view(m, H)
    root_c = torch.from_numpy(raw[first + rows * page:first + rows * page + m * H * 4].view(np.float32)).view(m, H)
    assert m * H * 4 > page and root_h.data_ptr() % page == 0
    out = dict(n_levels=torch.zeros(1, dtype=torch.int32, pin_memory=True), n_roots=torch.zeros(1, dtype=torch.int32, pin_memory=True),
               root_ids=torch.zeros(m, dtype=torch.int32, pin_memory=True), root_h=root_h, root_c=root_c)
    cudart = torch.cuda.cudart()
    assert int(cudart.cudaHostRegister(root_h.data_ptr(), page, 0)) == 0
    try:
        model.forward_host(*host, max_roots=m, out=out)
        assert int(out["n_roots"][0]) == f.n_trees
        np.testing.assert_array_equal(root_h[:f.n_trees].numpy(), good["root_h"].numpy())
    except binding.TreeLSTMError as err:
        assert err.code == binding.ERR_CUDA
    finally:
        torch.cuda.synchronize()
        assert int(cudart.cudaHostUnregister(root_h.data_ptr())) == 0
    again = model.forward_host(*host, max_roots=f.n_trees)
    np.testing.assert_array_equal(again["root_h"].numpy(), good["root_h"].numpy())


def test_bounded_waits_time_out_cleanly():
    """failure detection without a fault: a wait on a flag that nothing sets ends by its cycle limit,
    the status word says TIMEOUT, and the context keeps working afterwards"""
    w = fg.make_workload("tiny8", 0)
    ref = util.oracle_forward_cached("tiny8", 0)
    model = util.make_model(w.params, "fp32")
    model.set_option(binding.OPT_WAIT_LIMIT_CYCLES, 200)          # 200 * 1024 cycles, about 0.1 ms
    first_ok, status1, second_ok, status2 = model.selftest_waits()
    assert first_ok == 0 and status1 == binding.ERR_TIMEOUT
    assert second_ok == 0 and status2 == binding.ERR_TIMEOUT
    model.set_option(binding.OPT_WAIT_LIMIT_CYCLES, 1 << 20)
    res = util.gpu_forward(model, w.forest, binding.PERSISTENT)
    assert util.max_abs(res["h"], ref["h"]) < util.TOL["fp32"]


@pytest.mark.parametrize("H,E", [(33, 7), (170, 20), (200, 12), (96, 300)])
def test_fp32_persistent_odd_and_large_hidden_sizes(H, E):
    """hidden sizes that end in a partial 16-unit slice (33), odd sizes (scalar operand fetch), sizes
    whose weight slice still fits in shared memory (170) and sizes where it does not (200: the kernel
    streams the weights as in per-level mode); both modes against the oracle, and against each other"""
    rng = np.random.default_rng(H * 1000 + E)
    params = fg.draw_params(rng, H, E, 60, emb_dist="uniform", emb_scale=0.5, w_scale=0.3 / np.sqrt(H / 16))
    forest = fg.random_forest(rng, 40, 1, 30, 60)      # wide leaf wavefront (64-row tiles) and narrow ones
    forest, _ = fg.permute_node_ids(forest, rng)
    model = util.make_model(params, "fp32")
    h, c, _ = orc.forward_recursive(forest.left, forest.right, forest.token, params.emb, params.W, params.b)
    for flags in (binding.PER_LEVEL, binding.PERSISTENT):
        res = util.gpu_forward(model, forest, flags)
        assert util.max_abs(res["h"], h) < util.TOL["fp32"]
        assert util.max_abs(res["c"], c) < util.TOL["fp32"]


@pytest.mark.parametrize("kind", ["threshold", "permuted", "64 levels", "65 levels", "4200 levels", "single leaves", "largest", "beyond"])
def test_schedule_of_one_cluster(kind):
    """forests that one cluster schedules: the smallest, shuffled ids (every link crosses CTAs), one to three sorting
    passes, ids that fill the last CTA's range partly, the largest forest and the first one beyond it; roots in order"""
    rng = np.random.default_rng(21)
    params = fg.draw_params(rng, 2, 2, 50, emb_dist="uniform", emb_scale=0.1, w_scale=0.1)
    cap = 16 * 8192
    if kind in ("largest", "beyond"):          # chains of 3 nodes, built directly: left leaf, right leaf, their caller
        n = cap - cap % 3 + (3 if kind == "beyond" else 0)
        k = np.arange(n, dtype=np.int32)
        inner = k % 3 == 2
        forest = fg.Forest(np.where(inner, k - 2, -1).astype(np.int32), np.where(inner, k - 1, -1).astype(np.int32),
                           np.where(inner, -1, k % 50).astype(np.int32), k[inner], k // 3)
    elif kind == "single leaves":
        forest = fg.forest_from_shapes([None] * 4097, rng, 50)
    elif kind.endswith("levels"):
        depth = int(kind.split()[0])
        forest = fg.concat_forests([fg.random_forest(rng, 70, 40, 60, 50), fg.forest_from_shapes([fg.left_chain_shape(depth)], rng, 50)])
    else:
        forest = fg.random_forest(rng, 75, 20, 36, 50)
        forest = fg.concat_forests([forest, fg.forest_from_shapes([None] * (4096 - forest.n_nodes), rng, 50)]) if forest.n_nodes < 4096 else forest
        if kind == "permuted":
            forest, _ = fg.permute_node_ids(forest, rng)
    status, _, level, order, off = orc.schedule(forest.left, forest.right)
    model = util.make_model(params, "fp32")
    res = util.gpu_forward(model, forest, binding.PERSISTENT)
    util.check_schedule(res, dict(level=level, order=order, level_offset=off), forest.n_nodes)
    roots = model.roots(forest.n_trees)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(roots["root_ids"].cpu().numpy(), np.sort(forest.roots))


def test_malformed_forests_on_the_scheduling_cluster():
    """two callers for one node, a cycle, a child out of range, a bad token: the same codes as on any other path"""
    rng = np.random.default_rng(22)
    params = fg.draw_params(rng, 4, 4, 50, emb_dist="uniform", emb_scale=0.1, w_scale=0.1)
    base = fg.random_forest(rng, 120, 30, 50, 50)
    inner = np.flatnonzero(base.left >= 0)
    model = util.make_model(params, "fp32")

    def code(change):
        arrays = [base.left.copy(), base.right.copy(), base.token.copy()]
        change(*arrays)
        with pytest.raises(binding.TreeLSTMError) as err:
            model.forward(*[util.to_dev(a) for a in arrays], flags=binding.PERSISTENT)
        return err.value.code

    def twice(l, r, t): l[inner[7]] = l[inner[900]]
    def cycle(l, r, t):                        # top -> p -> q becomes top -> q's old child, and p and q point at each other
        top = next(k for k in inner[::-1] if l[k] >= 0 and l[l[k]] >= 0 and l[l[l[k]]] >= 0)
        p, q = l[top], l[l[top]]
        l[top], l[q] = l[q], p
    def out_of_range(l, r, t): r[inner[3]] = base.n_nodes
    def token(l, r, t): t[np.flatnonzero(base.left < 0)[-1]] = 50
    assert code(twice) == code(out_of_range) == binding.ERR_INVALID_FOREST
    assert code(cycle) == binding.ERR_INVALID_FOREST
    assert code(token) == binding.ERR_TOKEN_OUT_OF_RANGE
    util.gpu_forward(model, base, binding.PERSISTENT)


@pytest.mark.parametrize("H,E,kind", [(32, 320, "leaves"), (33, 321, "leaves"), (31, 5, "half"), (150, 319, "most"), (64, 643, "half"), (1, 1, "leaves")])
def test_fp32_leaves_at_the_limits_of_their_tiles(H, E, kind):
    """the leaves' kernel: 64 leaves, 33 to 48 and at most 32 of them among 64 consecutive ids, contractions of one, of exactly one
    full, of just over one and of three loads of the operands, slices of 32 units with one unit more or less"""
    rng = np.random.default_rng(H + E)
    params = fg.draw_params(rng, H, E, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.1)
    shapes = {"leaves": [None] * 193, "half": [fg.balanced_shape(32)] * 3 + [None], "most": [None, fg.left_chain_shape(4), None] * 25}[kind]
    forest = fg.forest_from_shapes(shapes, rng, 60)
    res = util.gpu_forward(util.make_model(params, "fp32"), forest, binding.PERSISTENT)
    h, c, _ = orc.forward_recursive(forest.left, forest.right, forest.token, params.emb, params.W, params.b)
    assert util.max_abs(res["h"], h) < util.TOL["fp32"] and util.max_abs(res["c"], c) < util.TOL["fp32"]


@pytest.mark.parametrize("kind", ["one node", "one climb each", "one node more", "longer than a cluster's lists", "deeper than the tables"])
def test_fp32_lists_from_the_leaves_kernel(kind):
    """the clusters' lists, planned beside the leaves: a lone leaf, as many nodes as the planning CTA climbs from at once (3 x 512) and one
    tree more, lists that are longer than a cluster's share of the workspace and more depths than the tables hold (the clusters then plan
    for themselves); ids in no order, the same states twice"""
    rng = np.random.default_rng(14)
    params = fg.draw_params(rng, 20, 9, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.1)
    sentences = [fg.random_split_shape(rng, int(k)) for k in rng.integers(2, 40, size=30)]
    base = fg.forest_from_shapes(sentences, rng, 60).n_nodes
    shapes = {"one node": [None], "one climb each": sentences + [None] * (1536 - base), "one node more": sentences + [None] * (1537 - base),
              "longer than a cluster's lists": sentences[:5] + [fg.left_chain_shape(600)] + [None] * 400,
              "deeper than the tables": [fg.left_chain_shape(1500)] + [fg.left_chain_shape(3)] * 200}[kind]
    forest = fg.forest_from_shapes(shapes, rng, 60)
    forest, _ = fg.permute_node_ids(forest, rng)
    order = orc.schedule(forest.left, forest.right)[3]
    h, c, _ = orc.forward_iterative(forest.left, forest.right, forest.token, params.emb, params.W, params.b, order)
    model = util.make_model(params, "fp32")
    first, again = (util.gpu_forward(model, forest, binding.PERSISTENT) for _ in range(2))
    assert util.max_abs(first["h"], h) < util.TOL["fp32"] and util.max_abs(first["c"], c) < util.TOL["fp32"]
    assert np.array_equal(first["h"], again["h"]) and np.array_equal(first["c"], again["c"])


@pytest.mark.parametrize("precision", ["fp32", "bf16"])
@pytest.mark.parametrize("n_trees", [1, 30, 300])
def test_forests_that_kernels_ahead_of_the_call_write(precision, n_trees):
    """the scheduler comes up while the launch ahead of it ends, here kernels that overwrite the forest's arrays in place (one forest, then
    another of the same size) with no wait by the host: every call sees its own forest; schedulers of one CTA, of a cluster, beside tree clusters"""
    rng = np.random.default_rng(15)
    params = fg.draw_params(rng, 40, 24, 100, emb_dist="normal", emb_scale=0.3, w_scale=0.1)
    sizes = rng.integers(2, 40, size=n_trees)
    forests = [fg.forest_from_shapes([fg.random_split_shape(rng, int(k)) for k in sizes], rng, 100) for _ in range(2)]
    model = util.make_model(params, precision)
    refs = [util.gpu_forward(model, f, binding.PERSISTENT) for f in forests]
    sources = [[util.to_dev(a) for a in (f.left, f.right, f.token)] for f in forests]
    arrays = [torch.zeros_like(a) for a in sources[0]]
    results = []
    for call in range(12):
        for to, a in zip(arrays, sources[call % 2]):
            torch.mul(a, 1, out=to)
        results.append(model.forward(*arrays, check=False))
    assert model.status_sync() == binding.OK
    for call, out in enumerate(results):
        for key in ("h", "c", "level", "order"):
            np.testing.assert_array_equal(out[key].cpu().numpy(), refs[call % 2][key])


def test_calls_go_to_the_current_stream():
    device, other = torch.cuda.current_device(), torch.cuda.Stream()
    assert binding._stream() == binding._public_raw_stream(device) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(other):
        assert binding._stream() == binding._public_raw_stream(device) == other.cuda_stream


@pytest.mark.parametrize("shapes", ["two chains", "a chain among sentences", "single leaves"])
def test_fp32_lists_of_more_nodes_than_climb_at_once(shapes):
    """forests beyond the 1536 nodes that the planning CTA climbs from: depths and roots by pointer jumping, ids in no order"""
    rng = np.random.default_rng(15)
    params = fg.draw_params(rng, 20, 9, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.15, n_classes=0)
    shapes = {"two chains": [fg.left_chain_shape(1025), fg.left_chain_shape(1000)], "single leaves": [None] * 1700,
              "a chain among sentences": [fg.left_chain_shape(200)] + [fg.random_split_shape(rng, int(k)) for k in rng.integers(2, 40, size=60)]}[shapes]
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 60), rng)
    order = orc.schedule(forest.left, forest.right)[3]
    h, c, _ = orc.forward_iterative(forest.left, forest.right, forest.token, params.emb, params.W, params.b, order)
    res = util.gpu_forward(util.make_model(params, "fp32"), forest, binding.PERSISTENT)
    assert util.max_abs(res["h"], h) < util.TOL["fp32"] and util.max_abs(res["c"], c) < util.TOL["fp32"]


@pytest.mark.parametrize("save", [0, binding.SAVE_FOR_BACKWARD])
@pytest.mark.parametrize("H,kind", [(150, "chain 86"), (150, "chain 200"), (256, "balanced 256"), (24, "random 120"), (24, "chain 1100"), (20, "chain 8192"), (64, "three long")])
def test_fp32_lists_of_one_or_a_few_longer_trees_are_planned_ahead(H, kind, save):
    """one cluster's lists may hold the whole forest, and one tree's depths are all there are: no cluster plans for itself behind the leaves
    (trace build: that would leave a stamp), and the states are the oracle's"""
    rng = np.random.default_rng(16)
    params = fg.draw_params(rng, H, 9, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.7 / np.sqrt(H), n_classes=3)
    shape, _, k = kind.partition(" ")
    shapes = {"chain": lambda: [fg.left_chain_shape(int(k))], "balanced": lambda: [fg.balanced_shape(int(k))], "random": lambda: [fg.random_split_shape(rng, int(k))],
              "three": lambda: [None, fg.left_chain_shape(150), fg.random_split_shape(rng, 200), fg.random_split_shape(rng, 3)]}[shape]()
    forest, _ = fg.permute_node_ids(fg.forest_from_shapes(shapes, rng, 60), rng)
    model = util.make_model(params, "fp32", variant="trace")
    model._workspace(forest.n_nodes, bool(save)).zero_()
    res = util.gpu_forward(model, forest, binding.PERSISTENT | save)
    setup = trace.read_trace(model, 0)[trace.LEVELS - 1]
    assert setup[2] > 0 and setup[5] == 0                                 # (lists there; no child table of the cluster's own)
    order = orc.schedule(forest.left, forest.right)[3]
    h, c, _ = orc.forward_iterative(forest.left, forest.right, forest.token, params.emb, params.W, params.b, order)
    assert util.max_abs(res["h"], h) < util.TOL["fp32"] and util.max_abs(res["c"], c) < util.TOL["fp32"]


@pytest.mark.parametrize("leaves", [16, 17, 20, 21, 28, 29, 32, 33])
def test_fp32_leaves_of_one_cta(leaves):
    """as many leaves as a warp's rows hold, and one more"""
    rng = np.random.default_rng(17)
    params = fg.draw_params(rng, 33, 321, 60, emb_dist="normal", emb_scale=0.3, w_scale=0.1)
    forest = fg.forest_from_shapes([None] * leaves, rng, 60)
    h, c, _ = orc.forward_recursive(forest.left, forest.right, forest.token, params.emb, params.W, params.b)
    res = util.gpu_forward(util.make_model(params, "fp32"), forest, binding.PERSISTENT)
    assert util.max_abs(res["h"], h) < util.TOL["fp32"] and util.max_abs(res["c"], c) < util.TOL["fp32"]
