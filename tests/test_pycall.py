"""Argument conversion of the calls that go through native code; nothing reaches the device here."""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

from paper_2412_14838_b200 import binding, build


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    binding.load()


def test_lists_of_tensors_arrays_and_addresses_reach_the_library():
    t, n = torch.zeros(8), np.zeros(8, dtype=np.float32)
    for items in ([t] * 3, [n, t.data_ptr(), None], (t,) * 100, []):
        with pytest.raises(binding.DkvError) as e:       # a NULL context: refused after the conversion
            binding.dkv_run_prefill_pass(0, items, items, items, items, items, 0)
        assert e.value.code == binding.DKV_ERR_INVALID_ARG
    with pytest.raises(binding.DkvError):
        binding.dkv_decode_attend(0, 0, 1, 1, [t], [t], [t], [t], stream=0)


@pytest.mark.parametrize("bad", [3, [object()], ["x"]])
def test_what_has_no_address_is_refused(bad):
    with pytest.raises(TypeError):
        binding.dkv_compact_all(0, 1, bad, [torch.zeros(4)], 0)


def test_a_configuration_passes_by_address():
    cfg = binding.make_config(4, 8, 2, 64, 1, 16, 16, 5, 64, 128, 2)       # S = ws: refused on the host
    with pytest.raises(binding.DkvError) as e:
        binding.dkv_score_static(cfg, torch.zeros(4), torch.zeros(4), torch.zeros(4), ctypes.c_void_p(0).value or 0)
    assert e.value.code == binding.DKV_ERR_INVALID_ARG


# Stands in for the library in a child process: how many of the DKV_MAX_LAYERS addresses it may read are not NULL.
STAND_IN = """
int dkv_run_prefill_pass(void* ctx, const void* const* q, const void* const* k, const void* const* v, void* const* kb, void* const* vb,
                         void* stream) {
  int n = 0;
  for (int i = 0; i < 128; ++i) n += q[i] != 0;
  return n;
}
"""
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def stand_in(tmp_path):
    (tmp_path / "stand_in.c").write_text(STAND_IN)
    lib = str(tmp_path / "stand_in.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", lib, str(tmp_path / "stand_in.c")], check=True)
    return lib


def test_lists_of_any_length_end_in_nulls(stand_in):
    code = ("from paper_2412_14838_b200 import binding as B; B.load()\n"
            "print([B._native().run_prefill_pass(0, [8] * n, [], [], [], [], 0) for n in (0, 1, 64, 65, 100, 127, 128, 200)])")
    # fresh memory is filled with a pattern, so that an entry that was never written is not NULL by chance
    env = dict(os.environ, LD_PRELOAD=stand_in, MALLOC_PERTURB_="90", PYTHONMALLOC="malloc")
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=env, capture_output=True, text=True, check=True)
    assert res.stdout.strip() == "[0, 1, 64, 65, 100, 127, 128, 128]"


def test_a_tensor_subclass_gives_its_own_address(stand_in):
    code = """
import torch
from paper_2412_14838_b200 import binding as B; B.load()
class Elsewhere(torch.Tensor):
    def data_ptr(self): return 0
class Plain(torch.Tensor): pass
t = torch.zeros(4)
items = [t, t.as_subclass(Elsewhere), t.as_subclass(Plain), torch.nn.Parameter(t), t.as_subclass(Elsewhere)]
print(B._native().run_prefill_pass(0, items, [], [], [], [], 0))
"""
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=stand_in), capture_output=True, text=True, check=True)
    assert res.stdout.strip() == "3"


def test_a_program_without_torch_makes_the_same_calls(stand_in):
    code = f"""
import sys
sys.modules["torch"] = None                                   # "import torch" fails
import ctypes, numpy as np
from paper_2412_14838_b200 import binding as B
def raises(kind, call):
    try: call()
    except kind as e: return getattr(e, "code", 0)
    raise AssertionError(kind)
B.load()
a = np.zeros(4, dtype=np.float32)
cfg = B.make_config(4, 8, 2, 64, 1, 16, 16, 5, 64, 128, 2)     # S = ws: refused on the host
refused = [lambda: B.dkv_decode_attend(0, 0, 1, 1, [a], [a], [a.ctypes.data], [a], stream=0), lambda: B.dkv_reset(0, 0),
           lambda: B.dkv_run_prefill_pass_host(0, [a], [a], [a], [a], [None], None), lambda: B.dkv_score_static(cfg, a, a, a, 0),
           lambda: B.dkv_memcpy_to_host(0, a, 8, a.nbytes, 0), lambda: B.dkv_rebudget(0, np.int64(1), stream=0)]
assert [raises(B.DkvError, c) for c in refused] == [B.DKV_ERR_INVALID_ARG] * len(refused)
raises(OverflowError, lambda: B.dkv_select_topk(0, 2**32, stream=0))
raises(TypeError, lambda: B.dkv_reset(0))                      # no stream, no torch whose current one to take
raises(TypeError, lambda: B.dkv_compact_all(0, 1, ["x"], [a], 0))
seen = []
library = ctypes.CDLL({stand_in!r}).dkv_run_prefill_pass           # the converted list as the library sees it
for n in (0, 1, 127, 128, 200):
    seen.append(library(None, B._argument(ctypes.POINTER(ctypes.c_void_p), [8] * n)))
assert seen == [0, 1, 127, 128, 128], seen
"""
    subprocess.run([sys.executable, "-c", code], cwd=ROOT, check=True)


@pytest.mark.parametrize("value", [2**31, 2**32, 2**32 + 1, -2**31 - 1, 2**70])
def test_an_integer_that_does_not_fit_is_refused(value):
    t = torch.zeros(4)
    for call in (lambda: binding.dkv_select_topk(0, value, stream=0), lambda: binding.dkv_rebudget(0, value, stream=0),
                 lambda: binding.dkv_decode_attend(0, 0, 1, value, [t], [t], [t], [t], stream=0)):
        with pytest.raises(OverflowError):
            call()
    for fits in (2**31 - 1, -2**31):
        with pytest.raises(binding.DkvError):                # reaches the library, which refuses the NULL context
            binding.dkv_select_topk(0, fits, stream=0)


def test_the_native_half_belongs_to_one_torch_version(monkeypatch, tmp_path):
    built = []
    note = tmp_path / "note"
    monkeypatch.setattr(build, "PYCALL_TORCH", str(note))
    monkeypatch.setattr(build, "_build_pycall", lambda verbose: (built.append(1), note.write_text(build.torch_version())))
    note.write_text("1.0.0")                                   # linked with another version: rebuilt, and only then
    build.build()
    build.build()
    assert built == [1]
    note.write_text("1.0.0")
    monkeypatch.setattr(binding, "_lib", None)
    monkeypatch.setattr(binding, "_call", None)
    with pytest.raises(RuntimeError, match="linked with torch 1.0.0"):
        binding.load()
