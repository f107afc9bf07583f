"""The standalone tempering and resampling steps' workspace: no more than the
grouping writes, exactly that much suffices, and a byte less is refused."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 4096, 16384])
@pytest.mark.parametrize("M", [1, 20, 100])
def test_workspace_is_what_is_used(n, M):
    import torch
    from paper_2109_00661_gb300 import _lib
    lib = _lib.load()
    size = int(lib.aem_smc_workspace_bytes(n, M))
    assert size <= 4 * (n + (M + 1) + M) + 3 * 63  # order, offsets and counts, each rounded up to 64 bytes
    g = torch.Generator(device="cuda").manual_seed(n + M)
    ll = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * 10
    model = torch.randint(0, M, (n,), generator=g, device="cuda", dtype=torch.int32)
    u = torch.randint(0, 1 << 40, (M,), generator=g, device="cuda", dtype=torch.int64)
    d, done = torch.zeros(1, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    inc, W = torch.zeros(M, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    anc = torch.full((n,), -1, dtype=torch.int32, device="cuda")
    buf = torch.full((size + 256,), 0x5A, dtype=torch.uint8, device="cuda")
    assert buf.data_ptr() % 64 == 0
    rw = (ll.data_ptr(), model.data_ptr(), n, M, 0.0, 0.5, 60, d.data_ptr(), done.data_ptr(), inc.data_ptr(),
          W.data_ptr(), buf.data_ptr())
    rs = (W.data_ptr(), model.data_ptr(), n, M, u.data_ptr(), anc.data_ptr(), buf.data_ptr())
    stream = torch.cuda.current_stream().cuda_stream
    assert lib.aem_reweight(*rw, size - 1, stream) == -1 and lib.aem_resample_systematic(*rs, size - 1, stream) == -1
    assert lib.aem_reweight(*rw, size, stream) == 0 and lib.aem_resample_systematic(*rs, size, stream) == 0
    torch.cuda.synchronize()
    assert torch.all(buf[size:] == 0x5A)
    assert torch.all((anc >= 0) & (anc < n)) and torch.all(model[anc.long()] == model)
