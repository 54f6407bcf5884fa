"""Argument checks of named launch plans, before any CUDA call: 2 values per thread at N = 16 and 32
are accepted as part of an FP64 plan (with the instances per block) and refused otherwise."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import _build, cme


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    cme.load()


def refused(N, **kw):
    try:
        cme.Batch([cme.Instance(N, np.ones(N), np.zeros(N), 1.0, 0.5, 1.0, 0.0)], **kw).close()
    except cme.CmeError as e:      # without a GPU, creation ends at the first CUDA call
        return e.code == -1
    return False


@pytest.mark.parametrize("N", [16, 32])
def test_two_values_per_thread_at_small_n(N):
    assert refused(N, radix=2)
    assert not refused(N, radix=2, inst_per_cta=4, cluster=1, persistent=1)
    assert refused(N, radix=2, inst_per_cta=4, precision=cme.FP32)
    assert refused(8, radix=2, inst_per_cta=4)
