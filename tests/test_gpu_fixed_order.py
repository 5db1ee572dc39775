"""The pipelined methods give the recorded results bit for bit (see _fixed_order.py)."""
import json

import pytest

import _fixed_order as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(lib):
    import torch
    from paper_1511_07226_gb300 import pfk
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("recorded on 152 SMs")
    return pfk.Context(0)


@pytest.mark.parametrize("name", list(F.CASES))
def test_recorded_bits(ctx, name):
    assert F.summary(F.solve_case(ctx, name)) == json.load(open(F.GOLDEN))[name]
