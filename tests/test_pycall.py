"""Argument conversion of the calls that go through native code; nothing reaches the device here."""
import ctypes

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
