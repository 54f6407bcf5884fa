"""Every launch plan that cme_batch_plan returns can be named in cme_batch_create's options, and gives
the same plan and the same bits again."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import cme

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [cme.FP64, cme.FP32])
@pytest.mark.parametrize("integ", [cme.RK4IP, cme.STRANG])
@pytest.mark.parametrize("N,count", [(4, 3), (8, 3), (16, 1), (16, 7), (16, 5000), (32, 1), (32, 9),
                                     (32, 3000), (64, 1), (64, 2500), (128, 3), (256, 3), (512, 3),
                                     (1024, 3), (2048, 3), (4096, 3), (4096, 120)])
def test_returned_plan_can_be_named(N, count, integ, prec):
    rng = np.random.default_rng(N)
    one = [cme.Instance(N, np.ones(N), np.zeros(N), 1.0, 0.5, 1.5, 1.0,
                        0.3 * rng.standard_normal((N, 2)).view(complex)[:, 0] / np.sqrt(N))
           for _ in range(3)]
    insts = [one[i % 3] for i in range(count)]
    chosen = cme.Batch(insts, precision=prec, integrator=integ)
    plan = {k: v for k, v in chosen.plan(0).items() if k != "N"}
    named = cme.Batch(insts, precision=prec, integrator=integ, **plan)
    assert {k: v for k, v in named.plan(0).items() if k != "N"} == plan
    for b in (chosen, named):
        b.step(1e-3, 2)
    np.testing.assert_array_equal(chosen.get_state(), named.get_state())
