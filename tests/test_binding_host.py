"""Host logic of the binding, with a stand-in for torch."""
import types

import pytest

from paper_1509_04953_gb300 import evp


@pytest.mark.parametrize("has_raw_call", [True, False])
def test_stream_handle_with_and_without_the_private_call(has_raw_call):
    cuda = types.SimpleNamespace(current_device=lambda: 3,
                                 current_stream=lambda: types.SimpleNamespace(cuda_stream=0x5eed + 3))
    core = types.SimpleNamespace()
    if has_raw_call:
        core._cuda_getCurrentRawStream = lambda device: 0x5eed + device
    assert evp._stream(types.SimpleNamespace(_C=core, cuda=cuda)) == 0x5eed + 3
