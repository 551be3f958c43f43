"""A plan that leaves the sum-row tile after its batch was built: the batch's work
list is not its any more, and binding says so."""
import numpy as np
import pytest

import oracle
import paper_2311_05341_gb300 as dd
from paper_2311_05341_gb300 import _lib
from paper_2311_05341_gb300 import batch as ddb
from synth import channel_freqs, filterbank

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _need_cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def test_binding_refuses_a_retiled_plan():
    freqs = channel_freqs(1500.0, 300.0, 640)
    step = 0.2 * 64e-6 / oracle.delay_coeff(freqs[-1], 1500.0)
    ranges = [(0.0, 200 * step, step, 1)]
    beams = [ddb.BeamSpec(freqs, 1500.0, 64e-6, ranges, "u8", 9000)] * 2
    runner = ddb.BatchRunner(beams, autotune=False, graph=False)
    assert runner.plans[1].run_kernel(0, 8900, scratch=False) == ("sum-rows", False)
    runner.plans[1].set_tile(0, 4)
    with pytest.raises(dd.DDError) as err:
        runner.bind()
    assert err.value.status == _lib.DD_ERR_INVALID_ARG
    runner.plans[1].set_tile(0, "pattern")
    runner.bind()
    x = filterbank(np.uint8, 640, 9000, 9900, 128, 40)
    for t in runner.inputs:
        t[:, :9000].copy_(torch.from_numpy(x))
    runner.run()
    runner.status()
    ref = oracle.forward(x, freqs, 1500.0, 64e-6, ranges)[0]
    for i in range(2):
        np.testing.assert_array_equal(runner.planes(i)[0].cpu().numpy(), ref)
