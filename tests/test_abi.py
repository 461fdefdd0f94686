"""CPU checks of the C-ABI boundary: the library builds, loads, exports every declared symbol, and its host-side
argument validation answers without touching a device."""
import ctypes
import os
import re

import pytest

from paper_2609_20888_b200 import binding as eb
from paper_2609_20888_b200 import build as ebuild

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    ebuild.build()
    return eb.load()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "eta.h")).read()
    declared = set(re.findall(r"^(?:int|size_t|const char\*)\s+(eta_\w+)\s*\(", header, flags=re.M))
    assert declared, "no declarations found in include/eta.h"
    assert declared == set(eb.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), f"{name} declared in eta.h but not exported"


def _desc(**kw):
    base = dict(batch=2, n_q_heads=8, n_kv_heads=2, head_dim=128, block_size=64, t_cap=4096, nb_cap=64,
                k_stride_b=2 * 4096 * 128, k_stride_h=4096 * 128, k_stride_t=128,
                v_stride_b=2 * 4096 * 128, v_stride_h=4096 * 128, v_stride_t=128)
    base.update(kw)
    return eb.CacheDesc(**base)


def test_workspace_bytes_and_validation(lib):
    n = eb.eta_workspace_bytes(_desc())
    assert n > 0 and n % 256 == 0
    # grows with the block capacity, not with anything else
    assert eb.eta_workspace_bytes(_desc(t_cap=8192, nb_cap=128)) > n
    sz = ctypes.c_size_t(0)
    for bad, code in [(_desc(head_dim=96), -2), (_desc(block_size=48), -2), (_desc(n_q_heads=6), -2),
                      (_desc(n_q_heads=7), -1), (_desc(batch=0), -1), (_desc(k_stride_t=100), -2),
                      (_desc(nb_cap=8), -1)]:
        assert lib.eta_workspace_bytes(ctypes.byref(bad), ctypes.byref(sz)) == code
    assert lib.eta_workspace_bytes(None, ctypes.byref(sz)) == -1
    assert lib.eta_workspace_bytes(ctypes.byref(_desc()), None) == -1


def test_null_and_inconsistent_arguments_are_rejected_before_any_launch(lib):
    d, p = _desc(), eb.DecodeParams().c()
    null = ctypes.c_void_p(None)
    one = ctypes.c_void_p(256)          # never dereferenced on the host
    assert lib.eta_build_block_summaries(ctypes.byref(d), null, one, one, one, 0, null) == -1
    assert lib.eta_append_summary(ctypes.byref(d), one, null, one, one, 0, null) == -1
    assert lib.eta_predict_threshold(1, 8, 128, null, one, one, one, null) == -1
    assert lib.eta_predict_threshold(0, 8, 128, one, one, one, one, null) == -1
    assert lib.eta_score_dual(ctypes.byref(d), None, one, one, one, one, one, null) == -1
    # both tau and head_const, then neither
    args = [ctypes.byref(d), ctypes.byref(p), one, one, one, one, one, one]
    tail = [one, one, null, null, one, 1 << 30, null]
    assert lib.eta_decode(*args, one, one, *tail) == -1
    assert lib.eta_decode(*args, null, null, *tail) == -1
    # misaligned workspace, too-small workspace
    assert lib.eta_decode(*args, one, null, one, one, null, null, ctypes.c_void_p(264), 1 << 30, null) == -3
    assert lib.eta_decode(*args, one, null, one, one, null, null, one, 16, null) == -3
    # misaligned K
    args_bad = list(args)
    args_bad[3] = ctypes.c_void_p(260)
    assert lib.eta_decode(*args_bad, one, null, *tail) == -2
    bad = eb.DecodeParams(rescue_window=0).c()
    args2 = [ctypes.byref(d), ctypes.byref(bad)] + args[2:]
    assert lib.eta_decode(*args2, one, null, *tail) == -1


def test_kernel_attributes_are_remembered_per_device(lib):
    """cudaFuncSetAttribute results hold per (device, kernel): the library's bookkeeping must ask again on a second
    device, ask again for more shared memory, not ask twice for the same, and never remember a failure.  Host-only
    self-check with made-up device ordinals and a recording setter; 0 = every expectation held."""
    lib.eta_selftest_kernel_attr_table.restype = ctypes.c_int
    assert lib.eta_selftest_kernel_attr_table() == 0


def test_status_text(lib):
    assert lib.eta_strerror(0) == b"ok"
    assert b"workspace" in lib.eta_strerror(-3)
    assert lib.eta_decode_kernel_count() >= 1


def test_binding_refuses_cpu_tensors(lib):
    import torch
    K = torch.zeros((1, 2, 128, 128), dtype=torch.bfloat16)
    d = eb.cache_desc(K, K, 8, 64)
    ms = torch.zeros((1, 2, 2, 2, 128), dtype=torch.float16)
    mn = torch.zeros((1, 2, 2), dtype=torch.float32)
    with pytest.raises(eb.EtaError):
        eb.eta_build_block_summaries(d, K, torch.zeros(1, dtype=torch.int32), ms, mn)


def test_step_calls_check_their_tensors():
    """The compiled marshalling refuses what the binding refuses: host tensors, other types, things that are no tensors."""
    import pytest
    import torch

    from paper_2609_20888_b200 import binding as eb
    eb.load()
    K = torch.zeros((1, 1, 64, 64), dtype=torch.bfloat16)
    f, i = torch.zeros(4), torch.zeros(1, dtype=torch.int32)
    desc = eb.cache_desc(K, K, 1, 64)
    with pytest.raises(eb.EtaError, match="K must be a CUDA tensor"):
        eb.eta_append_summary(desc, K, i, f, f)
    with pytest.raises(TypeError):
        eb.eta_append_summary(desc, 17, i, f, f)
    with pytest.raises(TypeError):
        eb.eta_append_summary(i.numpy(), K, i, f, f)
    with pytest.raises(eb.EtaError, match="q must be a CUDA tensor"):
        eb.eta_predict_threshold(torch.zeros((1, 1, 64), dtype=torch.bfloat16), f, f, f)
    with pytest.raises(RuntimeError):          # invalid argument; without a GPU, no stream to call it on
        eb.eta_decode(desc, eb.DecodeParams(), None, None, None, None, None, None, None, None, None, None, None)
    with pytest.raises(AttributeError):
        eb.eta_decode(desc, object(), None, None, None, None, None, None, None, None, None, None, None)


def test_the_signature_of_a_step_call_does_not_hang_on_its_arguments():
    """None for a page table, a descriptor or parameters, and False for a workspace, are refused; none of them selects another
    signature for the same entry point."""
    eb.load()
    d, p, none = _desc(), eb.DecodeParams(), [None] * 10
    for call in (lambda: eb.eta_append_summary_paged(d, None, None, None, None, None),
                 lambda: eb.eta_decode_paged(d, None, p, *none, None),
                 lambda: eb.eta_append_summary(None, None, None, None, None),
                 lambda: eb.eta_decode(None, p, *none, None),
                 lambda: eb.eta_decode_static(None, p, *none),
                 lambda: eb.eta_decode(d, p, *none, False),
                 lambda: eb.eta_decode_paged(d, eb.PageTable(), p, *none, False)):
        with pytest.raises(TypeError):
            call()
    with pytest.raises(AttributeError):
        eb.eta_decode(d, None, *none, None)


def test_step_calls_take_no_other_structure_of_the_same_size():
    eb.load()
    none = [None] * 4
    wide = ctypes.create_string_buffer(ctypes.sizeof(eb.CacheDesc))
    two = (ctypes.c_int64 * 2)()
    assert ctypes.sizeof(two) == ctypes.sizeof(eb.PageTable)
    for call in (lambda: eb.eta_append_summary(wide, *none),
                 lambda: eb.eta_append_summary(bytes(wide), *none),
                 lambda: eb.eta_append_summary_paged(_desc(), two, *none),
                 lambda: eb.eta_decode(wide, eb.DecodeParams(), *none, *none, None, None, None)):
        with pytest.raises(TypeError):
            call()


def test_step_calls_read_parameters_as_ctypes_does():
    """The marshalled structure has the bytes of DecodeParams.c(): integers modulo 2^32, no truncated floats, whatever an
    override of c() returns."""
    import numpy as np
    eb.load()

    class Doubled(eb.DecodeParams):
        def c(self):
            return eb.Params(2 * self.z, self.a, self.beta, self.scale, self.lwb, self.rescue_window, self.flags)

    native = eb._native
    for kw in (dict(), dict(z=0.1, a=-2, beta=1e300, scale=np.float32(0.3)), dict(lwb=np.int64(3), rescue_window=64, flags=5),
               dict(lwb=True, flags=-1), dict(lwb=2 ** 32 + 1, rescue_window=2 ** 31), dict(rescue_window=-(2 ** 40) - 7)):
        for cls in (eb.DecodeParams, Doubled):
            assert native.params(cls(**kw)) == bytes(cls(**kw).c()), (cls, kw)
    for kw in (dict(lwb=2.7), dict(rescue_window=64.0), dict(flags=np.float32(1)), dict(lwb=None), dict(z="1"),
               dict(rescue_window=float("nan"))):
        with pytest.raises(TypeError):
            eb.DecodeParams(**kw).c()
        with pytest.raises(TypeError):
            native.params(eb.DecodeParams(**kw))
        with pytest.raises(TypeError):
            eb.eta_decode(_desc(), eb.DecodeParams(**kw), *[None] * 10, None)


def test_only_the_step_calls_need_the_compiled_marshalling(monkeypatch):
    """A missing (or unloadable) _eta_torch is an error of the calls that go through it, loudly; the library and the other entry
    points work without it."""
    import sys
    package = eb.__name__.rsplit(".", 1)[0]
    monkeypatch.setitem(sys.modules, package + "._eta_torch", None)        # an import of it fails
    monkeypatch.delattr(package + "._eta_torch", raising=False)
    monkeypatch.setattr(eb, "_native", None)
    monkeypatch.setattr(eb, "_lib", None)
    assert eb.eta_workspace_bytes(_desc()) > 0
    assert eb.eta_static_scratch_bytes() == 8 << 20
    with pytest.raises(eb.EtaError, match="_eta_torch is missing"):
        eb.eta_append_summary(_desc(), None, None, None, None)
    with pytest.raises(eb.EtaError, match="_eta_torch is missing"):
        eb.eta_decode(_desc(), eb.DecodeParams(), *[None] * 10, None)


def test_the_marshalling_is_rebuilt_for_another_torch(monkeypatch):
    """It links against torch's C++ interface: one that was built for another version is not current, whatever its date."""
    import torch
    ebuild.build_torch_module()
    assert ebuild.torch_module_is_current()
    monkeypatch.setattr(torch, "__version__", "0.0.0")
    assert not ebuild.torch_module_is_current()
