"""The compiled host side of the step calls (_binding): what it refuses, with the texts of the Python checks, and what it reads from its
arguments.  Nothing here reaches a GPU: every call is refused by a check or by the library (no context)."""
import ctypes as C

import numpy as np
import pytest
import torch

import __graft_entry__
from paper_2511_21699_b200 import api


@pytest.fixture(scope="module")
def host():
    __graft_entry__.build()
    return api._host()


class _Stream:
    cuda_stream = 0


def _tree(t):
    return dict(tokens=t, parent=t, depth=t, mask=t, n_nodes=t)


def test_tensors_that_are_refused(host):
    h, s = C.c_void_p(None), _Stream()
    cpu = torch.zeros(4, 4, dtype=torch.int32)
    for call in (lambda x: host.update(h, x, cpu, cpu, s), lambda x: host.reset(h, x, s), lambda x: host.draft_tree(h, x, cpu, _tree(cpu), s),
                 lambda x: host.accept(h, _tree(x), None, None, _tree(x), s), lambda x: host.kv_commit(h, x, x, x, x, x, x, x, x, s),
                 lambda x: host.tree_attn(h, x, x, x, x, x, x, x, x, x, x, None, 0, 0.0, s)):
        for bad in (cpu, cpu.t(), [1, 2], np.zeros(4, np.int32), "x", 3):
            with pytest.raises((api.CachebackError, TypeError), match="expected a contiguous CUDA tensor|subscript|indices"):
                call(bad)


def test_logits_that_are_refused(host):
    h, s = C.c_void_p(None), _Stream()
    t = torch.zeros(2, 4, dtype=torch.int32)
    for dtype in (torch.float16, torch.float64, torch.int32):
        with pytest.raises(api.CachebackError, match="logits must be float32 or bfloat16"):
            host.accept(h, _tree(t), torch.zeros(2, 4, 8, dtype=dtype), None, {}, s)
    for x in (torch.zeros(2, 4, 8), torch.zeros(8, 8), torch.zeros(2, 4, 16)[..., ::2]):
        with pytest.raises(api.CachebackError, match="uniform row stride"):
            host.accept_update_draft_tree(h, _tree(t), x, t, t, _tree(t), {}, s)


def test_calls_without_a_context_reach_the_library_and_come_back_as_errors(host):
    for h in (C.c_void_p(None), None):                          # None: a context that was closed
        with pytest.raises(api.CachebackError, match="cb_reset failed: invalid argument"):
            host.reset(h, None, _Stream())


def test_arguments_of_the_wrong_number_or_kind(host):
    t = torch.zeros(2, 4, dtype=torch.int32)
    with pytest.raises(TypeError, match="expected 5 arguments"):
        host.update(C.c_void_p(None), t, t)
    with pytest.raises(AttributeError):
        host.reset(C.c_void_p(None), None, object())             # not a stream
    with pytest.raises(KeyError):
        host.accept(C.c_void_p(None), {}, None, None, {}, _Stream())


def test_module_is_built_again_for_another_torch_or_interpreter(monkeypatch, tmp_path):
    """File times say nothing of what the module was compiled against."""
    import os
    import sys
    import types
    from paper_2511_21699_b200 import build
    calls = []

    def compiler(cmd, **kw):
        calls.append(cmd)
        open(cmd[cmd.index("-o") + 1], "w").close()
    monkeypatch.setattr(build, "SO_BINDING", str(tmp_path / "_binding.so"))
    monkeypatch.setattr(build.subprocess, "check_call", compiler)
    for want in (1, 1):                                         # built once, then found as it is
        build.build_binding()
        assert len(calls) == want
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".other")
    build.build_binding()
    build.build_binding()
    assert len(calls) == 2
    tag = types.SimpleNamespace(**dict(vars(sys.implementation), cache_tag="cpython-other"))
    monkeypatch.setattr(build.sys, "implementation", tag)
    build.build_binding()
    assert len(calls) == 3 and os.path.exists(build.SO_BINDING)
