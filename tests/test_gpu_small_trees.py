"""Trees of at most 32 nodes on the tensor-core path (their own kernel, commit and verification in one pass over the state)
against the fp64 oracle: both tile sizes at their edges, every form of the commit, ragged and padded packing."""
import numpy as np
import pytest

from paper_2607_06763_b200 import synth
from tests.test_gpu_padded import PaddedDevice, _assert_outputs, _oracle_commit, _oracle_verify

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tl(cuda_device):
    from tests import gdn_testlib
    return gdn_testlib


def _tree(rng, kind, n):
    if kind == "chain":
        return synth.tree_chain(min(n, 16))
    if kind == "star":
        return synth.tree_star(n)
    return synth.tree_geo(rng, n)


@pytest.mark.parametrize("out_dtype", [synth.BF16, synth.F32])
@pytest.mark.parametrize("sizes", [(1, 2, 8, 9, 15, 16), (1, 16, 17, 24, 31, 32)])
def test_step_and_verification_of_small_trees(tl, sizes, out_dtype):
    """One call per shape of tree; accepted paths of 0, 1, 7, 8, 9 and 16 nodes (one and two tiles of steps)."""
    from tests.test_gpu_parity import _fused_case
    rng = np.random.default_rng(77)
    prev_trees = [synth.tree_chain(16) for _ in sizes]
    paths = [np.arange(n, dtype=np.int32) for n in (0, 1, 7, 8, 9, 16)]
    prev = synth.random_case(701, prev_trees, 2, 6, 128, 128, synth.BF16, out_dtype, paths=paths, name="prev")
    for i, kind in enumerate(("geo", "chain", "star")):
        new = synth.random_case(710 + i, [_tree(rng, kind, n) for n in sizes], 2, 6, 128, 128, synth.BF16, out_dtype, name="new")
        _fused_case(tl, prev, new, f"{kind} {sizes}")
        dc = tl.DeviceCase(new)
        before = dc.S0.clone()
        assert dc.verify() == 0 and dc.device_status() == 0
        assert bool((dc.S0 == before).all())
        tl.assert_close_per_head(dc.o_host(), tl.oracle_verify(new), new.node_offsets, f"verify {kind}", bf16_out=tl.is_bf16_out(new))


@pytest.mark.parametrize("raw_gates", [False, True])
@pytest.mark.parametrize("t_pad,sizes", [(16, (16, 3)), (19, (19, 1)), (32, (32, 17))])
def test_padded_step_of_small_trees(tl, t_pad, sizes, raw_gates):
    import paper_2607_06763_b200 as gdn
    rng = np.random.default_rng(t_pad)
    prev = synth.padded_case(720, [synth.tree_chain(16), synth.tree_chain(10)], 3, 40, raw_gates,
                             paths=[np.arange(11, dtype=np.int32), np.arange(5, dtype=np.int32)])
    new = synth.padded_case(721, [synth.tree_geo(rng, n) for n in sizes], 3, t_pad, raw_gates)
    dp, dn = PaddedDevice(prev), PaddedDevice(new)
    S = dp.S0.clone()
    rc = gdn.gdn_tree_commit_verify_padded(dn.shape, new.n_trees, raw_gates, S, prev.t_pad, dp.k, dp.v, dp.g_in, dp.beta_in, dp.parent,
                                           dp.n_nodes, dp.path, dp.path_len, dn.q, dn.k, dn.v, dn.g_in, dn.beta_in, dn.parent,
                                           dn.n_nodes, dn.o, dn.status)
    assert rc == 0 and dn.status_value() == 0
    S_ref = _oracle_commit(prev, prev.S0.astype(np.float64))
    tl.assert_state_close(S.cpu().numpy().astype(np.float64), S_ref, what="state")
    _assert_outputs(tl, dn, _oracle_verify(new, S_ref), f"padded step, {t_pad} rows")


@pytest.mark.parametrize("T", [16, 32])
def test_small_trees_are_as_exact_as_large_ones(tl, T):
    """fp32 outputs, error in the norm: q' and the state are bf16 hi + lo, as for trees of 64 nodes (2.7e-6 there; the terms
    dropped are 2^-17 of a factor each)."""
    w = synth.random_case(730, [_tree(np.random.default_rng(s), "geo", T) for s in range(8)], 4, 8, 128, 128, synth.BF16, synth.F32)
    dc = tl.DeviceCase(w)
    assert dc.verify() == 0 and dc.device_status() == 0
    ref = tl.oracle_verify(w)
    assert np.linalg.norm(dc.o_host() - ref) <= 2.0 ** -17 * np.linalg.norm(ref)


@pytest.mark.parametrize("raw_gates", [False, True])
@pytest.mark.parametrize("t_pad,sizes,n_layers,out_dtype", [(1, (1,), 2, synth.BF16), (16, (16, 9), 3, synth.F32), (16, tuple(range(1, 17)) * 3, 1, synth.BF16),
                                                            (32, (32,), 3, synth.BF16), (31, (17, 31, 2), 2, synth.F32)])
def test_planned_verification_of_small_trees(tl, t_pad, sizes, n_layers, out_dtype, raw_gates):
    """Trees found in the plan's list (more than a warp of records among them); an empty tree has none, a plan of another
    shape is refused on the device."""
    import torch
    import paper_2607_06763_b200 as gdn
    from tests.test_gpu_padded import _plan
    rng = np.random.default_rng(sum(sizes) + t_pad)
    w = synth.padded_case(740 + t_pad + len(sizes), [synth.tree_geo(rng, n) for n in sizes], n_layers, t_pad, raw_gates, out_dtype=out_dtype)
    d = PaddedDevice(w)
    plan = _plan(d, w)
    call = lambda plan: gdn.gdn_tree_verify_planned(d.shape, w.n_trees, raw_gates, d.S0, d.q, d.k, d.v, d.g_in, d.beta_in, plan, d.o, d.status)
    assert call(plan) == 0 and d.status_value() == 0
    _assert_outputs(tl, d, _oracle_verify(w), f"planned, {t_pad} rows")
    d.n_nodes[0] = 0
    plan = _plan(d, w)
    d.o.fill_(7.0)
    assert call(plan) == 0 and d.status_value() == 0
    o = d.o_host()
    assert np.all(o[:: w.n_trees] == 7.0) and (w.n_trees == 1 or np.any(o[1] != 7.0))
    d.o.fill_(7.0)
    assert call(torch.zeros_like(plan)) == 0 and d.status_value() == -10
    assert np.all(d.o_host() == 7.0)


def _units(limit):
    """(units, nodes a tree may have) at both sides of the rules of the small-tree kernel, from the number of SMs."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    return {"four parts, 16": (sms // 4, 16), "four parts, 32": (sms // 4, 32), "two parts, first, 16": (sms // 4 + 1, 16),
            "two parts, last, 16": (sms // 2, 16), "two parts, 32": (sms // 2, 32), "one part, 16": (sms // 2 + 1, 16),
            "one part, 32": (sms // 2 + 1, 32), "last of 32": (2 * sms, 32), "first beyond 32": (2 * sms + 1, 32),
            "last at three": (3 * sms, 16), "first at four": (3 * sms + 1, 16), "last at four": (4 * sms, 16),
            "three again": (4 * sms + 1, 16), "four, 8 nodes": (4 * sms + 1, 8), "many of 32": (5 * sms, 32)}[limit]


@pytest.mark.parametrize("out_dtype", [synth.BF16, synth.F32])
@pytest.mark.parametrize("packing", ["ragged", "padded"])
@pytest.mark.parametrize("limit", ["four parts, 16", "four parts, 32", "two parts, first, 16", "two parts, last, 16", "two parts, 32",
                                   "one part, 16", "one part, 32", "last of 32", "first beyond 32", "last at three", "first at four",
                                   "last at four", "three again", "four, 8 nodes", "many of 32"])
def test_step_on_both_sides_of_every_rule(tl, limit, packing, out_dtype):
    """One head a slot, so that the units can be counted out; paths of 0, 1, 7, 8, 9 and 16 nodes, trees of all sizes, one of them
    empty, one with a parent[] that points forward, one path that is not a chain.  The state that the small-tree kernel commits is
    held to fp32 rounding (see test_commit_is_as_exact_in_every_form)."""
    import paper_2607_06763_b200 as gdn
    from oracle import gdn_oracle as orc
    slots, T = _units(limit)
    rng = np.random.default_rng(slots + T)
    lens = [(0, 1, 7, 8, 9, 16)[i % 6] for i in range(slots)]
    sizes = [T] + [1 + (5 * i) % T for i in range(1, slots)]
    trees = [synth.tree_geo(rng, n) if n > 1 else np.array([-1], np.int32) for n in sizes]
    prev_trees = [synth.tree_chain(16)] * slots
    paths = [np.arange(n, dtype=np.int32) for n in lens]
    paths_ok = list(paths)
    paths[5], paths_ok[5] = np.array([0, 2], np.int32), np.zeros(0, np.int32)
    bad = next(i for i in range(8, slots) if sizes[i] > 2)
    if packing == "ragged":
        trees[4] = np.zeros(0, np.int32)
        prev, prev_ok = (synth.random_case(750, prev_trees, 1, 1, 128, 128, synth.BF16, out_dtype, paths=p) for p in (paths, paths_ok))
        new = synth.random_case(751, trees, 1, 1, 128, 128, synth.BF16, out_dtype)
        dp, dn = tl.DeviceCase(prev), tl.DeviceCase(new)
        dn.parent[int(new.node_offsets[bad]) + 1] = 2
        S = dp.S0.clone()
        rc = gdn.gdn_tree_commit_verify(dn.shape, S, dp.k, dp.v, dp.g, dp.beta, dp.parent, dp.node_offsets, dp.path, dp.path_offsets,
                                        dn.q, dn.k, dn.v, dn.g, dn.beta, dn.parent, dn.node_offsets, dn.o, dn.ws, dn.ws_bytes, dn.status)
        S_ref = tl.oracle_commit(prev_ok)
        o_ref = orc.verify(S_ref, *(new.f64(n) for n in ("q", "k", "v", "g", "beta")), new.parent, new.node_offsets, new.scale)
        rows = [slice(int(a), int(b)) for a, b in zip(new.node_offsets, new.node_offsets[1:])]
        untouched, status = 0.0, dn.device_status
    else:
        prev, prev_ok = (synth.padded_case(752, prev_trees, 1, 16, True, h_qk=1, h_v=1, paths=p, out_dtype=out_dtype) for p in (paths, paths_ok))
        new = synth.padded_case(753, trees, 1, T, True, h_qk=1, h_v=1, out_dtype=out_dtype)
        dp, dn = PaddedDevice(prev), PaddedDevice(new)
        dn.n_nodes[4] = 0
        dn.parent[bad, 1] = 2
        S = dp.S0.clone()
        rc = gdn.gdn_tree_commit_verify_padded(dn.shape, new.n_trees, True, S, 16, dp.k, dp.v, dp.g_in, dp.beta_in, dp.parent, dp.n_nodes,
                                               dp.path, dp.path_len, dn.q, dn.k, dn.v, dn.g_in, dn.beta_in, dn.parent, dn.n_nodes,
                                               dn.o, dn.status)
        S_ref = _oracle_commit(prev_ok, prev.S0.astype(np.float64))
        o_ref = _oracle_verify(new, S_ref)
        rows = [(i, slice(0, 0 if i == 4 else sizes[i])) for i in range(slots)]
        untouched, status = 7.0, dn.status_value
    assert rc == 0 and status() in (-7, -9)
    o, S = dn.o_host(), S.cpu().numpy().astype(np.float64)
    tl.assert_state_close(S, S_ref, what="state")
    large = limit in ("first beyond 32", "many of 32")
    if not large:   # (the kernel of 64-node tiles takes the path step by step, scaled: a rounding of the state each)
        assert np.linalg.norm(S - S_ref) <= 7.2e-8 * np.linalg.norm(S_ref)
    assert np.array_equal(S[5], prev.S0[5]) and np.array_equal(S[0], prev.S0[0])
    # value by value (seven rows at a time: too few for the norm-wise bound on bf16 rounding, a statistical one, which would be asked
    # of 600 slots one by one), and that bound over all slots
    err = ref = 0.0
    for i, r in enumerate(rows):
        if i == bad:
            assert np.all(o[r] == untouched)
        elif i != 4:
            err, ref = err + ((o[r] - o_ref[r]) ** 2).sum(), ref + (o_ref[r] ** 2).sum()
            for j in range(0, sizes[i], 7):
                x, y = o[r][j:j + 7], o_ref[r][j:j + 7]
                tl.assert_close_per_head(x, y, np.array([0, len(x)]), f"{limit}, {packing}, slot {i}", bf16_out=out_dtype == synth.BF16)
    # fp32 outputs: a bf16 rounding is off by 1.66e-3 in the norm, a pair by 1.66e-3 of its low term; the pairs of the state, those of q' and
    # the low terms' product, which is dropped, make sqrt(3) 1.66e-3^2 = 4.8e-6 at most (64-node tiles have a third pair and two products)
    assert err <= (tl.TOL_BF16_NORMWISE if out_dtype == synth.BF16 else 2.0 ** -17 if large else 4.8e-6) ** 2 * ref
    if packing == "padded":
        assert all(np.all(o[i, (0 if i in (4, bad) else sizes[i]):] == 7.0) for i in range(slots))


@pytest.mark.parametrize("t_pad", [5, 16])
def test_planned_verification_of_many_small_trees(tl, t_pad):
    """300 trees in each of two layers, some empty, some rejected when the plan is built: the records of the others stand in the list
    in any order, and every slot finds its own tree."""
    import paper_2607_06763_b200 as gdn
    from tests.test_gpu_padded import _plan
    rng = np.random.default_rng(t_pad)
    sizes = rng.integers(1, t_pad + 1, size=300)
    w = synth.padded_case(760 + t_pad, [synth.tree_geo(rng, int(n)) if n > 1 else np.array([-1], np.int32) for n in sizes], 2, t_pad, False, h_qk=1, h_v=2)
    d = PaddedDevice(w)
    empty, bad = {0, 31, 32, 150, 299}, {1, 33, 298} | {int(i) for i in range(0, 300, 37)}
    bad = {i for i in bad - empty if sizes[i] > 2}
    for i in empty:
        d.n_nodes[i] = 0
    for i in bad:
        d.parent[i, 1] = 2
    plan = _plan(d, w)
    assert d.status_value() == -7
    d.status.zero_()
    assert gdn.gdn_tree_verify_planned(d.shape, w.n_trees, False, d.S0, d.q, d.k, d.v, d.g_in, d.beta_in, plan, d.o, d.status) == 0
    assert d.status_value() == 0
    o, ref = d.o_host(), _oracle_verify(w)
    for s in range(w.n_slots):
        t = s % 300
        n = 0 if t in empty | bad else int(sizes[t])
        assert np.all(o[s, n:] == 7.0)
        for j in range(0, n, 7):   # (see above)
            tl.assert_close_per_head(o[s, j:min(n, j + 7)], ref[s, j:min(n, j + 7)], np.array([0, min(n, j + 7) - j]), f"slot {s}", bf16_out=True)


@pytest.mark.parametrize("at", [0, 3, 9])
@pytest.mark.parametrize("g_strong", [-3000.0, -np.inf])
@pytest.mark.parametrize("slots,T", [(1, 16), (2, 16), (4, 16), (15, 16), (1, 32), (2, 32), (4, 32)])
def test_step_behind_a_strong_decay_on_the_path(tl, slots, T, g_strong, at):
    """One strong decay (alpha = 0 at the last) on accepted paths of weak ones (32 heads: four, two and one CTA per unit, three and four
    per SM): the steps behind it keep their precision, and so do the outputs on the committed state."""
    from tests.test_gpu_parity import _fused_case
    rng = np.random.default_rng(T)
    prev = synth.random_case(770, [synth.tree_chain(16)] * slots, 2, 32, 128, 128, synth.BF16, synth.F32,
                             paths=[np.arange(16 if i % 2 == 0 else 7, dtype=np.int32) for i in range(slots)])
    prev.g[:] = synth.f32_to_bf16_bits(np.float32([-0.0101]))[0]
    prev.g[at::16] = synth.f32_to_bf16_bits(np.float32([g_strong]))[0]
    new = synth.random_case(771, [synth.tree_geo(rng, T) for _ in range(slots)], 2, 32, 128, 128, synth.BF16, synth.F32)
    _fused_case(tl, prev, new, f"step behind g = {g_strong}")


@pytest.mark.parametrize("T", [16, 32])
def test_trees_deeper_than_max_depth_are_rejected_one_by_one(tl, T):
    """max_depth = 8: chains of 9 nodes are reported and write nothing, those of 8 and the others are verified, alone and fused."""
    import paper_2607_06763_b200 as gdn
    trees = [synth.tree_chain(8), synth.tree_chain(9), synth.tree_star(T), synth.tree_chain(9), np.array([-1], np.int32)]
    w = synth.random_case(772, trees, 2, 4, 128, 128, synth.BF16, synth.F32, paths=[np.zeros(0, np.int32)] * 5)
    ref = tl.oracle_verify(w)
    for fused in (False, True):
        dc = tl.DeviceCase(w, max_depth=8)
        dc.o.fill_(7.0)
        if fused:
            assert gdn.gdn_tree_commit_verify(dc.shape, dc.S0, dc.k, dc.v, dc.g, dc.beta, dc.parent, dc.node_offsets, dc.path, dc.path_offsets,
                                              dc.q, dc.k, dc.v, dc.g, dc.beta, dc.parent, dc.node_offsets, dc.o, dc.ws, dc.ws_bytes, dc.status) == 0
        else:
            assert dc.verify() == 0
        assert dc.device_status() == -8
        o = dc.o_host()
        for b in range(5):
            r = slice(int(w.node_offsets[b]), int(w.node_offsets[b + 1]))
            if b in (1, 3):
                assert np.all(o[r] == 7.0)
            else:
                tl.assert_close_per_head(o[r], ref[r], np.array([0, len(o[r])]), f"tree {b}")


@pytest.mark.parametrize("slots,T", [(1, 16), (2, 32), (5, 16), (5, 32)])
def test_captured_steps_of_small_trees(tl, slots, T):
    """Step, verification and (the same trees in the dense layout) planned verification in one graph: replayed, bit for bit what the
    calls give."""
    import torch
    import paper_2607_06763_b200 as gdn
    rng = np.random.default_rng(T)
    prev = synth.random_case(773, [synth.tree_chain(16)] * slots, 16, 32, 128, 128, synth.BF16, synth.BF16,
                             paths=[np.arange((9, 16, 3, 0, 8)[i], dtype=np.int32) for i in range(slots)])
    new = synth.random_case(774, [synth.tree_geo(rng, T) for _ in range(slots)], 16, 32, 128, 128, synth.BF16, synth.BF16)
    dp, dn = tl.DeviceCase(prev), tl.DeviceCase(new)
    S, o2, o3 = dp.S0.clone(), torch.zeros_like(dn.o), torch.zeros_like(dn.o)
    nodes = torch.full((slots,), T, dtype=torch.int32, device="cuda")
    plan = torch.zeros(gdn.gdn_tree_plan_bytes(dn.shape, slots), dtype=torch.uint8, device="cuda")

    def step(st):
        assert gdn.gdn_tree_commit_verify(dn.shape, S, dp.k, dp.v, dp.g, dp.beta, dp.parent, dp.node_offsets, dp.path, dp.path_offsets,
                                          dn.q, dn.k, dn.v, dn.g, dn.beta, dn.parent, dn.node_offsets, dn.o, dn.ws, dn.ws_bytes, dn.status, st) == 0
        assert gdn.gdn_tree_verify(dn.shape, S, dn.q, dn.k, dn.v, dn.g, dn.beta, dn.parent, dn.node_offsets, o2, dn.ws, dn.ws_bytes,
                                   dn.status, st) == 0
        assert gdn.gdn_tree_plan(dn.shape, slots, dn.parent, nodes, plan, dn.status, st) == 0
        assert gdn.gdn_tree_verify_planned(dn.shape, slots, False, S, dn.q, dn.k, dn.v, dn.g, dn.beta, plan, o3, dn.status, st) == 0

    step(torch.cuda.current_stream())
    assert dn.device_status() == 0
    S_ref = tl.oracle_commit(prev)
    tl.assert_state_close(S.cpu().numpy().astype(np.float64), S_ref, what="state")
    from tests.test_gpu_parity import dataclass_replace_S0
    ref = tl.oracle_verify(dataclass_replace_S0(new, S_ref))
    for o in (dn.o, o2, o3):
        tl.assert_close_per_head(o.float().cpu().numpy().astype(np.float64), ref, new.node_offsets, "outputs", bf16_out=True)
    eager = [x.clone() for x in (S, dn.o, o2, o3)]
    graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=side):
        step(torch.cuda.current_stream())
    for _ in range(3):
        S.copy_(dp.S0)
        for o in (dn.o, o2, o3):
            o.zero_()
        graph.replay()
        assert dn.device_status() == 0 and all(bool((a == b).all()) for a, b in zip((S, dn.o, o2, o3), eager))
