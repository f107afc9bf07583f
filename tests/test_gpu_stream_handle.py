"""Calls go to torch's current stream, with or without the release's raw stream handle."""
import pytest

from paper_2109_00661_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream_is_used(monkeypatch, raw):
    import torch
    import paper_2109_00661_gb300 as L
    if not raw:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    sysg = L.System(**I.system_kwargs("sounding-g20-f40-k120"))
    models = I.to_torch(I.random_models(8, seed=1), torch.float32)
    want = L.forward_f32(sysg, models)
    torch.cuda.synchronize()
    for stream in (torch.cuda.current_stream(), torch.cuda.Stream()):
        with torch.cuda.stream(stream):
            assert L._stream_ptr(None).value in ((stream.cuda_stream,) if stream.cuda_stream else (None, 0))
            got = L.forward_f32(sysg, models)
        stream.synchronize()
        assert torch.equal(got, want)
