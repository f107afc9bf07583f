"""The FP32 forward kernel's bounded wait for the next model, made to run out
(no poll at all): the timeout is recorded, the answer is waited for again, and
no model is lost."""
import pytest

from paper_2109_00661_gb300 import inputs as I

pytestmark = pytest.mark.gpu
ERR_TIMEOUT = -4


@pytest.mark.parametrize("name, lmax, P", [("sounding-g20-f40-k120", 3, 1300), ("sounding-g20-f40-k120", 8, 9000),
                                           ("forward-g30-f60-k200", 10, 2500)])
def test_a_claim_whose_wait_runs_out_is_still_answered(name, lmax, P):
    import torch
    import paper_2109_00661_gb300 as L
    sysg = L.System(**I.system_kwargs(name))
    models = I.to_torch(I.random_models(P, seed=P, lmax=lmax, layers_max=lmax), torch.float32)
    y, ref = torch.full((sysg.G,), 1e-9, dtype=torch.float64, device="cuda"), L.System(**I.system_kwargs(name))
    ref.set_forward_shape(lmax, 1)  # fixed order: no claims
    want = L.loglik_f32(ref, models, y, 1e-11, 0.03, want_gates=True)
    assert sysg.forward_shape(lmax, P) in (10, 11)
    assert L.system_status(sysg) == 0
    L.debug_bounded_wait(sysg, spins=1)
    try:
        got = L.loglik_f32(sysg, models, y, 1e-11, 0.03, want_gates=True)
        torch.cuda.synchronize()
        assert L.system_status(sysg) == ERR_TIMEOUT
        assert L.system_status(sysg) == 0  # read and cleared
    finally:
        L.debug_bounded_wait(sysg, spins=0)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    again = L.loglik_f32(sysg, models, y, 1e-11, 0.03, want_gates=True)
    assert torch.equal(again[0], want[0]) and torch.equal(again[1], want[1])
    assert L.system_status(sysg) == 0
