"""The native part of the Python binding: which file it is, and where it gets the current stream from."""
import sysconfig
import types

import pytest
import torch

from paper_2508_02558_b200 import binding as B
from paper_2508_02558_b200 import build as libbuild


def test_marshal_module_carries_the_abi_tag_of_this_python():
    libbuild.build()
    native = B.native()
    assert native.__file__ == B.MARSHAL_PATH == libbuild.MARSHAL
    assert B.MARSHAL_PATH.endswith("_marshal" + sysconfig.get_config_var("EXT_SUFFIX"))


@pytest.mark.parametrize("private", [True, False])
def test_current_stream_with_and_without_torchs_private_getters(private, monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda dev=None: types.SimpleNamespace(cuda_stream=1000 + dev))
    for name, value in (("_cuda_getDevice", lambda: 4), ("_cuda_getCurrentRawStream", lambda dev: 2000 + dev)):
        monkeypatch.setattr(torch._C, name, value, raising=False)
        if not private:
            monkeypatch.delattr(torch._C, name)
    raw, device = B._stream_getters()
    assert (device(), raw(device())) == ((4, 2004) if private else (3, 1003))
