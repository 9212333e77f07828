"""The binding's current-stream handle (lib.stream_ptr): torch's private shortcut
where it exists, the public Stream object where it does not."""
from types import SimpleNamespace

import pytest

from paper_2504_14494_gb300 import lib as L


@pytest.mark.parametrize("private", [True, False])
def test_handle_with_and_without_the_private_function(monkeypatch, private):
    c = SimpleNamespace(_cuda_getCurrentRawStream=lambda dev: 100 + dev) if private else SimpleNamespace()
    cuda = SimpleNamespace(current_device=lambda: 3,
                           current_stream=lambda: SimpleNamespace(cuda_stream=42))
    monkeypatch.setattr(L, "_torch_module", SimpleNamespace(_C=c, cuda=cuda))
    assert L.stream_ptr() == (103 if private else 42)
    assert L.stream_ptr(7) == 7 and L.stream_ptr(SimpleNamespace(cuda_stream=8)) == 8
