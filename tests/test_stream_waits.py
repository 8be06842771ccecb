"""Which torch streams a call with device inputs waits for (the streams faked: no GPU needed)."""
import types

import paper_1909_10690_gb300 as mi


def test_the_current_stream_of_every_device_with_an_input(monkeypatch):
    waited = []

    def current_stream(dev):
        return types.SimpleNamespace(synchronize=lambda: waited.append(dev))

    monkeypatch.setattr(mi, "_torch", lambda: types.SimpleNamespace(cuda=types.SimpleNamespace(current_stream=current_stream)))
    arg = lambda dev: types.SimpleNamespace(on_gpu=dev is not None, obj=types.SimpleNamespace(device=dev))  # noqa: E731
    mi._wait_for(arg(None), arg("cuda:0"), arg("cuda:1"), arg("cuda:0"), arg(None))
    assert waited == ["cuda:0", "cuda:1"]
