"""What the entry points launch, and in which order, without a GPU: the library's objects linked with ``fake_cudart.c`` in
place of the CUDA runtime.  No kernel runs."""
import ctypes
import os
import re
import shutil
import subprocess
import threading

import numpy as np
import pytest

import paper_2607_06763_b200 as gdn
from paper_2607_06763_b200 import binding, build

HERE = os.path.dirname(os.path.abspath(__file__))
A = 1 << 20   # an address that is aligned for everything; nothing is read there


@pytest.fixture(scope="module")
def fake_path(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("fake"))
    build.build_library()   # (the argument marshaller)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    flags = ["-gencode", "arch=compute_100a,code=compute_100a", "-O1", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler",
             "-fno-gnu-unique", "-I", os.path.join(build._ROOT, "include"), "-I", build.CSRC]
    objects = [os.path.join(d, os.path.basename(s)[:-3] + ".o") for s in build.sources()]
    jobs = [subprocess.Popen([nvcc] + flags + ["-c", "-o", o, s]) for s, o in zip(build.sources(), objects)]
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    fake = os.path.join(d, "fake.o")
    subprocess.check_call(["gcc", "-O1", "-fPIC", "-c", "-o", fake, os.path.join(HERE, "fake_cudart.c")])
    path = os.path.join(d, "libgdn_fake.so")
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", path] + objects + [fake])
    return path


class Fake:
    """A copy of the library of its own: everything a process keeps is as at its start."""
    n = 0

    def __init__(self, path):
        Fake.n += 1
        copy = f"{path}.{Fake.n}"
        shutil.copy(path, copy)
        self.lib = ctypes.CDLL(copy)
        self.lib.fake_log.restype = ctypes.c_char_p
        self.reset()

    def reset(self, fail_call=-1):
        self.lib.fake_reset(fail_call)

    def call(self, name, *args):
        return binding._call(ctypes.cast(getattr(self.lib, name), ctypes.c_void_p).value, *args)

    def count(self, name):
        return self.lib.fake_log().decode().split().count(name)

    def launches(self):
        return re.findall(r"\d((?:commit|verify|plan)_[a-z0-9_]*?kernel)(?=[EI])", self.lib.fake_log().decode())   # (mangled names)


def _shape(n_seq, T, in_dtype=1, d=128, h_v=32):
    return gdn.GdnShape(n_seq, h_v // 2, h_v, d, d, in_dtype, 1, 16, n_seq * T, T, 0.0883883)


def _fused(fake, s, S=A):
    ws = fake.lib.gdn_tree_workspace_bytes(ctypes.byref(s))
    return fake.call("gdn_tree_commit_verify", s, S, *[A] * 15, A, A, ws, A, 0)


def _fused_padded(fake, s, S=A):
    return fake.call("gdn_tree_commit_verify_padded", s, 1, 0, S, s.max_tree_nodes, *[A] * 17, A, 0)


FUSED = [
    (_fused, _shape(1, 64), A, ["commit_tile128_kernel", "verify_plain_kernel"]),
    (_fused_padded, _shape(1, 64), A, ["commit_tile128_kernel", "verify_plain_kernel"]),
    (_fused, _shape(48, 64), A, ["commit_verify_kernel"]),
    (_fused_padded, _shape(48, 64), A, ["commit_verify_kernel"]),
    (_fused, _shape(4, 256), A, ["commit_plan_kernel", "verify_plain_kernel"]),
    (_fused, _shape(4, 64, in_dtype=0), A, ["commit_generic_kernel", "verify_generic_small_kernel"]),
    (_fused, _shape(4, 100, d=64), A, ["plan_kernel", "commit_generic_kernel", "verify_generic_kernel"]),
    # trees of at most 32 nodes: one pass, as long as units or nodes are few
    (_fused, _shape(1, 16), A, ["verify_step_small_kernel"]),
    (_fused_padded, _shape(2, 16), A, ["verify_step_small_kernel"]),
    (_fused, _shape(48, 16), A, ["verify_step_small_kernel"]),
    (_fused_padded, _shape(4, 32), A, ["verify_step_small_kernel"]),
    (_fused, _shape(10, 32), A, ["commit_verify_kernel"]),
    # a state off a 32-byte boundary
    (_fused, _shape(1, 64), A + 16, ["commit_generic_kernel", "verify_generic_small_kernel"]),
    (_fused, _shape(48, 256), A + 16, ["plan_kernel", "commit_generic_kernel", "verify_generic_kernel"]),
]


@pytest.mark.parametrize("call,shape,S,kernels", FUSED, ids=range(len(FUSED)))
def test_fused_call_commits_only_once_the_verification_is_prepared(fake_path, call, shape, S, kernels):
    """The commit advances the state in place: where a CUDA call of the host path fails, short of a launch, the call must not
    have touched the state (or have gone through by another route: queries that only choose between routes)."""
    fake = Fake(fake_path)
    assert call(fake, shape, S) == 0 and fake.launches() == kernels
    n = fake.lib.fake_calls()
    assert n > 0
    for k in range(n):
        fresh = Fake(fake_path)
        fresh.reset(k)
        rc = call(fresh, shape, S)
        if rc == 0:
            assert fresh.launches() in (kernels, ["commit_verify_kernel"])
        else:
            assert rc == -6 and not any("commit" in x for x in fresh.launches()), f"call {k} of {n} failed behind the commit"


@pytest.mark.parametrize("units,T,form", [(1, 16, (16, 2, 4)), (37, 16, (16, 2, 4)), (38, 16, (16, 2, 2)), (74, 1, (16, 2, 2)), (75, 16, (16, 3, 1)),
                                          (444, 16, (16, 3, 1)), (445, 16, (16, 4, 1)), (592, 16, (16, 4, 1)), (593, 16, (16, 3, 1)),
                                          (593, 8, (16, 4, 1)), (37, 17, (32, 2, 4)), (74, 32, (32, 2, 2)), (75, 32, (32, 2, 1)), (296, 32, (32, 2, 1))])
def test_forms_of_the_step_of_small_trees(fake_path, units, T, form):
    """On 148 SMs: nodes of a tile, CTAs per SM and CTAs per unit of the kernel that a fused call takes."""
    fake = Fake(fake_path)
    s = gdn.GdnShape(units, 1, 1, 128, 128, 1, 1, 16, units * T, T, 0.0883883)
    assert _fused(fake, s) == 0
    n, ctas, parts = form
    assert f"verify_step_small_kernelILi{n}E13__nv_bfloat16Lb1ELi{ctas}ELb0ELi{parts}EE" in fake.lib.fake_log().decode()


@pytest.mark.parametrize("call,shape,S,kernels", FUSED, ids=range(len(FUSED)))
def test_shared_memory_limits_are_raised_in_every_context(fake_path, call, shape, S, kernels):
    """Limits raised in one context do not count in another one (after cudaDeviceReset, say): every launch has its own."""
    fake = Fake(fake_path)
    for context in (3, 3, 4, 3, 0):
        fake.lib.fake_context(ctypes.c_ulonglong(context))
        fake.reset()
        assert call(fake, shape, S) == 0 and fake.launches() == kernels, f"context {context}"


def test_static_scratch_is_found_in_every_context(fake_path):
    """The address of the library's scratch array belongs to a context: it is asked for in each, and once."""
    fake, s = Fake(fake_path), _shape(1, 100, d=32, h_v=4)
    for context, asked in ((3, 1), (3, 0), (4, 1), (4, 0), (5, 1)):
        fake.lib.fake_context(ctypes.c_ulonglong(context))
        fake.reset()
        assert fake.call("gdn_tree_verify_static", s, *[A] * 10, 0) == 0
        assert fake.launches() == ["plan_kernel", "verify_generic_kernel"] and fake.count("cudaGetSymbolAddress") == asked


def _fused_host(fake, s):
    """gdn_tree_commit_verify_host of trees of max_tree_nodes nodes, paths of one node (the arrays read on the host are real)."""
    nodes = np.arange(s.n_seq + 1, dtype=np.int32) * s.max_tree_nodes
    paths = np.arange(s.n_seq + 1, dtype=np.int32)
    arena = fake.lib.gdn_tree_commit_verify_host_arena_bytes(ctypes.byref(s), s.total_nodes, s.n_seq)
    return fake.call("gdn_tree_commit_verify_host", s, A, s.total_nodes, *[A] * 5, nodes, A, paths, s.n_seq, *[A] * 6, nodes, A, A,
                     arena, 0)


def test_host_buffer_pipeline_has_streams_in_every_context(fake_path):
    """The helper streams and events of the pipelined call belong to a context: each has its own, made once."""
    fake, s = Fake(fake_path), _shape(4, 64)
    for context, made in ((3, 2), (3, 0), (4, 2), (3, 0), (4, 0)):
        fake.lib.fake_context(ctypes.c_ulonglong(context))
        fake.reset()
        assert _fused_host(fake, s) == 0
        assert fake.launches() == ["commit_tile128_kernel", "verify_plain_kernel"] * 4 and fake.count("cudaStreamCreate") == made


def test_host_buffer_pipeline_is_one_thread_at_a_time(fake_path):
    """The calls of a context share its helper streams and events: an event that one thread has recorded is waited for by the
    same thread before another one records it again."""
    fake, s, rcs = Fake(fake_path), _shape(6, 64), []
    threads = [threading.Thread(target=lambda: rcs.append(_fused_host(fake, s))) for _ in range(3)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    who = [x for x in fake.lib.fake_log().decode().split() if x.startswith("record:")]
    assert rcs == [0] * 3 and len(who) == 3 * (2 + 2 * 6)
    assert sum(a != b for a, b in zip(who, who[1:])) == 2, "calls of several threads ran into one another"
