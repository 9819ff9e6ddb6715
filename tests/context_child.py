"""Run by test_calls_in_a_second_context: the host-buffer entry points in driver contexts made here, without torch."""
import ctypes
import os
import sys

import numpy as np

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import paper_2607_06763_b200 as gdn  # noqa: E402
from oracle import gdn_oracle as orc  # noqa: E402
from paper_2607_06763_b200 import synth  # noqa: E402

cuda = ctypes.CDLL("libcuda.so.1")


def check(rc):
    assert rc == 0, f"driver call failed: {rc}"


class Context:
    def __init__(self):
        self.handle, dev = ctypes.c_void_p(), ctypes.c_int()
        check(cuda.cuDeviceGet(ctypes.byref(dev), 0))
        check(cuda.cuCtxCreate_v2(ctypes.byref(self.handle), 0, dev))
        self.arena_bytes, self.arena = 64 << 20, ctypes.c_uint64()
        check(cuda.cuMemAlloc_v2(ctypes.byref(self.arena), ctypes.c_size_t(self.arena_bytes)))

    def use(self):
        check(cuda.cuCtxSetCurrent(self.handle))

    def destroy(self):
        check(cuda.cuCtxDestroy_v2(self.handle))


def run(ctx, w):
    """verify and commit of one workload, against the oracle."""
    ctx.use()
    s = gdn.GdnShape.from_workload(w)
    o = np.zeros((w.total_nodes, w.h_v, w.d_v), np.float32)
    rc = gdn.gdn_tree_verify_host(s, w.S0, w.q, w.k, w.v, w.g, w.beta, w.parent, w.node_offsets, o, ctx.arena.value,
                                  ctx.arena_bytes)
    assert rc == 0, gdn.gdn_status_string(rc)
    S = w.S0.copy()
    rc = gdn.gdn_tree_commit_host(s, S, w.k, w.v, w.g, w.beta, w.parent, w.node_offsets, w.path, w.path_offsets, len(w.path),
                                  ctx.arena.value, ctx.arena_bytes)
    assert rc == 0, gdn.gdn_status_string(rc)
    args = [w.f64(n) for n in ("S0", "q", "k", "v", "g", "beta")]
    o_ref = orc.verify(*args, w.parent, w.node_offsets, w.scale)
    S_ref = orc.commit(args[0], *args[2:], w.parent, w.node_offsets, w.path, w.path_offsets)
    assert np.abs(o - o_ref).max() <= 1e-4 * np.abs(o_ref).max()
    assert np.abs(S - S_ref).max() <= 1e-4 * np.abs(S_ref).max()


def main():
    check(cuda.cuInit(0))
    rng = np.random.default_rng(5)
    cases = [synth.random_case(1, [synth.tree_geo(rng, T) for T in sizes], 2, 4, 128, 128, dt, synth.F32)
             for dt in (synth.F32, synth.BF16) for sizes in ((60, 20), (100,))]
    first = Context()
    for w in cases:
        run(first, w)
    second = Context()
    for ctx in (second, first):
        for w in cases:
            run(ctx, w)
    first.destroy()
    second.destroy()
    third = Context()
    for w in cases:
        run(third, w)
    third.destroy()


main()
