"""The current stream's handle comes from torch's own query, or, in a torch build without
it, from the public current_stream()."""
import types

import paper_2202_12756_gb300 as fft3d


def _fake_torch(**private):
    stream = lambda index: types.SimpleNamespace(cuda_stream=1000 + index)
    return types.SimpleNamespace(_C=types.SimpleNamespace(**private), cuda=types.SimpleNamespace(current_stream=stream))


def test_public_query_serves_where_the_private_one_is_missing(monkeypatch):
    monkeypatch.setattr(fft3d, "_torch_module", _fake_torch())
    assert fft3d._raw_stream(3) == 1003


def test_private_query_is_used_where_there_is_one(monkeypatch):
    monkeypatch.setattr(fft3d, "_torch_module", _fake_torch(_cuda_getCurrentRawStream=lambda index: 2000 + index))
    assert fft3d._raw_stream(3) == 2003
