"""The launch shape a call takes: the recorded one, 0 included, whatever the
number of models; the rule's while none is recorded."""
import pytest

from paper_2109_00661_gb300 import F32_SHAPES
from paper_2109_00661_gb300 import inputs as I

pytestmark = pytest.mark.gpu

COUNTS = (1, 300, 700, 1500, 200000)  # at most two models per SM, one wave, more than are resident


@pytest.mark.parametrize("name", list(I.CONFIGS))
def test_a_recorded_shape_is_taken_for_every_batch(name):
    import torch
    import paper_2109_00661_gb300 as L
    sysg = L.System(**I.system_kwargs(name))
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    small, large = sysg.forward_shape(10, 2 * sms), sysg.forward_shape(10, 200000)
    assert small == 2 and large in (F32_SHAPES, F32_SHAPES + 1)
    assert sysg.forward_shape(10, 2 * sms + 1) == large - F32_SHAPES  # one wave: the fixed order
    for shape in range(F32_SHAPES):
        sysg.set_forward_shape(10, shape)
        assert [sysg.forward_shape(10, n) for n in COUNTS] == [shape] * len(COUNTS)
    assert sysg.forward_shape(9, 2 * sms) == 2  # another lmax: none recorded
    models = I.to_torch(I.random_models(2048, seed=3), torch.float32)
    shape, _ = sysg.autotune(models, repeats=1)
    assert [sysg.forward_shape(10, n) for n in COUNTS] == [shape] * len(COUNTS)


def test_forward_shape_refuses_what_is_out_of_range():
    import paper_2109_00661_gb300 as L
    sysg = L.System(**I.system_kwargs("sounding-g20-f40-k120"))
    for lmax, n in ((0, 1), (21, 1), (8, -1)):
        with pytest.raises(L.AEMError):
            sysg.forward_shape(lmax, n)
    for shape in (-1, F32_SHAPES):
        with pytest.raises(L.AEMError):
            sysg.set_forward_shape(8, shape)
