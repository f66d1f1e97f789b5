"""Host only: the binding's host module belongs to one interpreter and one torch, and calls do without it."""
import os
import sys

import pytest
import torch

from paper_2405_14917_b200 import binding, build


def test_the_file_is_named_after_interpreter_and_torch():
    name = os.path.basename(build.HOST_PATH)
    assert torch.__version__ in name and sys.implementation.cache_tag in name


@pytest.mark.parametrize("content", [None, b"not a shared object"])
def test_calls_do_without_a_host_module_that_cannot_be_loaded(tmp_path, monkeypatch, content):
    path = tmp_path / "slim_host.so"
    if content is not None:
        path.write_bytes(content)
    monkeypatch.setattr(binding, "HOST_PATH", str(path))
    monkeypatch.setattr(binding, "_host", None)
    with pytest.warns(UserWarning, match="host module"):
        binding.host()
    # the general path is reached (and refuses a tensor that is not on the device)
    x = torch.zeros((1, 128), dtype=torch.float16)
    with pytest.raises(TypeError):
        binding.mpq_gemv(x, x, [2], x, x, 16, x)
    assert binding.host().linear() is None and binding.host().run_set() is None
