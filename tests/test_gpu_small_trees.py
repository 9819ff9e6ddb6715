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
