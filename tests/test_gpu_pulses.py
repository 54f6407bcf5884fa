"""FP64 right-hand sides and steps of short pulses (flat and sech spectra at sixteen sizes over one
octave; bounds and reasons in test_fixed_bounds.py), where a transform's samples reach the fixed
point's limit: one-block shapes, clusters, and the four-step kernels, whose row with the peak of a
pulse at time 0 is a flat field of its own."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import cme
from test_fixed_bounds import (G0, KAPPA, SIGMA, ULP, pulses, rel, rhs_extended, rk4ip_extended,
                               strang_extended)

pytestmark = pytest.mark.gpu
PUMP = 0.5


def batch(fields, **kw):
    N = fields.shape[-1]
    return cme.Batch([cme.Instance(N, np.full(N, KAPPA), np.zeros(N), G0, 1.0, PUMP, SIGMA,
                                   np.fft.fftshift(D)) for D in fields], **kw)


def modes(flat, N):
    return np.fft.ifftshift(np.asarray(flat).reshape(-1, N), axes=-1)


def rhs_error(D, **kw):
    N = D.shape[-1]
    b = batch(D, **kw)
    want = rhs_extended(D)
    want[:, 0] += PUMP
    err = rel(modes(b.eval_rhs(), N), want)
    b.close()
    return err


@pytest.mark.parametrize("N,R", [(4, 4), (16, 8), (32, 8), (64, 8), (128, 16), (256, 8), (512, 8),
                                 (1024, 8), (2048, 8), (2048, 16), (4096, 8), (4096, 16)])
def test_rhs_of_short_pulses(N, R):
    err = rhs_error(pulses(N), radix=R, cluster=1)
    assert err.max() <= ULP * 4 * (np.log2(N) + 2), int(err.argmax())


@pytest.mark.parametrize("N,kw", [(16, {}), (32, {}), (64, {"radix": 8}), (128, {}),
                                  (512, {"radix": 8}), (1024, {}), (1024, {"radix": 4}),
                                  (4096, {"cluster": 1}), (256, {"radix": 8, "cluster": 2}),
                                  (2048, {"cluster": 4}), (4096, {"cluster": 8})])
@pytest.mark.parametrize("integ,step,phase", [(cme.RK4IP, rk4ip_extended, 0.2),
                                              (cme.STRANG, strang_extended, 0.2),
                                              (cme.STRANG, strang_extended, 5.0)])
def test_steps_of_short_pulses(N, kw, integ, step, phase):
    for D in np.moveaxis(pulses(N).reshape(16, -1, N), 1, 0):
        h = float(phase / (G0 * np.abs(np.fft.ifft(D) * N).max() ** 2))
        b = batch(D, integrator=integ, **kw)
        b.step(h, 1)
        err = rel(modes(b.get_state(), N), step(D, h, PUMP))
        b.close()
        assert err.max() <= ULP * 8 * (np.log2(N) + 4), int(err.argmax())


@pytest.mark.parametrize("logN", [13, 14, 16, 18])
def test_rhs_of_a_short_pulse_in_four_steps(logN):
    N = 1 << logN
    mu = np.fft.ifftshift(np.arange(N) - N // 2)
    size = 2.0 ** (np.arange(-8, 0) / 8)
    for width in (N / 64, N / 16, N / 4):
        D = size[:, None] / np.cosh(np.minimum(np.abs(mu / width), 300.0))
        err = rhs_error(D)
        assert err.max() <= ULP * 4 * (logN + 2), (width, int(err.argmax()))
