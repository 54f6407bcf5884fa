"""FP64 RK4IP steps in fixed point, on the device: the error of modes far below the pumped one (bounds
in test_fixed_bounds.py) with and without clusters, and instances that share a block."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import cme
from test_fixed_bounds import G0, KAPPA, SIGMA, combs, small_mode_errors

pytestmark = pytest.mark.gpu


def step(D, h, pump, n=1, **kw):
    N = D.shape[-1]
    b = cme.Batch([cme.Instance(N, np.full(N, KAPPA), np.zeros(N), G0, 1.0, pump, SIGMA,
                                np.fft.fftshift(d)) for d in D], **kw)
    b.step(h, n)
    got = np.fft.ifftshift(b.get_state().reshape(-1, N), axes=-1)
    b.close()
    return got


@pytest.mark.parametrize("N,kw", [(16, {}), (64, {}), (128, {}), (512, {}), (512, {"radix": 8}),
                                  (1024, {}), (4096, {"cluster": 1}), (2048, {"cluster": 2}),
                                  (2048, {"cluster": 8}), (4096, {"cluster": 2}),
                                  (4096, {"cluster": 4}), (4096, {"cluster": 8})])
def test_small_modes_of_an_rk4ip_step(N, kw):
    D = combs(N, np.random.default_rng(int(np.log2(N))), 128 if N < 1024 else 32)
    h = 1e-3 if N <= 128 else 5e-4 if N <= 512 else 2e-4
    fixed, plain = small_mode_errors(D, step(D, h, 1.5, **kw), h, 1.5)
    assert fixed <= 2 * plain


@pytest.mark.parametrize("N", [16, 64, 128])
def test_steps_of_one_block_scale_apart(N):
    """Instances that share a warp or a block end with the bits they have alone."""
    D = combs(N, np.random.default_rng(N), 6) * np.array([1, 1e-3, 30, 1e-200, 0, 1])[:, None]
    together = step(D, 1e-3, 1.5, 3, radix=8)
    for d, got in zip(D, together):
        np.testing.assert_array_equal(got, step(d[None], 1e-3, 1.5, 3, radix=8)[0])
