"""The native argument module belongs to one Python ABI, and the stream is found with torch's public interface alone."""
import sysconfig
import types

import torch

from paper_2510_25600_b200 import binding as P
from paper_2510_25600_b200 import build


def test_the_module_is_named_after_the_interpreter_that_built_it():
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert suffix != ".so" and build.MARSHAL.endswith("_marshal" + suffix)
    assert P._marshal.__file__ == build.MARSHAL


def test_the_current_stream_without_torchs_private_functions(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    assert P._stream_getter(types.SimpleNamespace())() == 77
    assert P._stream_getter(types.SimpleNamespace(_cuda_getCurrentRawStream=lambda d: 10 + d))() == 77
    assert P._stream_getter(types.SimpleNamespace(_cuda_getCurrentRawStream=lambda d: 10 + d, _cuda_getDevice=lambda: 3))() == 13
