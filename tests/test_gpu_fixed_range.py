"""The ends of the FP64 range in the fixed-point kernels: what is not finite is reported, by both
integrators, with and without clusters, and zeros stay zeros."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import cme

pytestmark = pytest.mark.gpu
PLANS = [(16, {}), (64, {"radix": 8}), (512, {}), (1024, {}), (4096, {"cluster": 1}),
         (2048, {"cluster": 4}), (4096, {"cluster": 8})]


def batch(N, D, A_in=0.7, **kw):
    return cme.Batch([cme.Instance(N, np.ones(N), np.zeros(N), 1.3, 0.5, A_in, 1.0, d) for d in D],
                     **kw)


@pytest.mark.parametrize("N,kw", PLANS)
@pytest.mark.parametrize("integ", [cme.RK4IP, cme.STRANG])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e155, 1e200])
def test_non_finite_steps_are_reported(N, kw, integ, bad):
    rng = np.random.default_rng(N)
    D = rng.standard_normal((3, N, 2)).view(complex)[..., 0] / np.sqrt(N)
    b = batch(N, D, integrator=integ, **kw)
    D[1, 1] = bad
    b.set_state(D.reshape(-1))
    b.step(1e-3, 1)
    assert list(b.status()) == [0, 1, 0]
    got = b.get_state().reshape(3, N)
    assert not np.isfinite(got[1]).any() and np.isfinite(got[[0, 2]]).all()


@pytest.mark.parametrize("N,kw", PLANS)
@pytest.mark.parametrize("integ", [cme.RK4IP, cme.STRANG])
def test_unpumped_zero_fields_stay_zero(N, kw, integ):
    D = np.zeros((3, N), complex)
    D[1, 1] = 1e-160
    b = batch(N, D, A_in=0.0, integrator=integ, **kw)
    b.step(1e-3, 3)
    got = b.get_state().reshape(3, N)
    assert list(b.status()) == [0, 0, 0]
    assert got[1, 1] != 0 and not np.delete(got[1], 1).any() and not got[[0, 2]].any()


def test_per_mode_kerr_batches_hold_no_stage_tables():
    """The fixed-point stages' propagator (16 bytes per mode) is held only where stages run on it: a
    batch with per-mode Kerr coefficients needs 8 bytes per mode for those and not more."""
    torch = pytest.importorskip("torch")
    N, count = 256, 256

    def held(kerr):
        insts = [cme.Instance(N, np.ones(N), np.zeros(N), 1.0, 0.5, 0.7, 1.0,
                              np.zeros(N, complex), None, kerr)] * count
        before = torch.cuda.memory_allocated()
        b = cme.Batch(insts)
        used = torch.cuda.memory_allocated() - before
        b.close()
        return used

    cme.use_torch_allocator()
    try:
        plain, kerr = held(None), held(np.linspace(0.9, 1.1, N))
    finally:
        cme.load().cme_set_allocator(cme.ALLOC_FN(), cme.FREE_FN(), None)
    assert 0 < kerr <= plain - 8 * N * count + 4096


@pytest.mark.parametrize("N", [16, 64, 512, 4096])
def test_gain_through_the_entry_point_without_allocation(N):
    """cme_rk4ip_noalloc cannot check kappa on the host: a gain of up to 1.2 per half step integrates as
    in FP64, and a larger one is reported by NaN, not by a finite field."""
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(N)
    D = rng.standard_normal((N, 2)).view(complex)[:, 0] / np.sqrt(N)
    h = 2e-3

    def run(kappa):
        dev = [torch.tensor(v, dtype=torch.float64, device="cuda")
               for v in (np.full(N, kappa), np.zeros(N), [1.3, 1.0, 0.5, 0.0, 1.0],
                         D.view(float).copy())]
        cme.rk4ip_noalloc(N, 1, h, 2, *(v.data_ptr() for v in dev),
                          torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        return dev[3].cpu().numpy().view(complex)

    L = np.clongdouble
    for kappa in (-1.0, -360.0):
        E = np.exp((L(-kappa / 2) - 1j) * L(h) / 2)
        x = np.fft.ifftshift(D).astype(L)

        def F(y):
            a = np.fft.ifft(y) * N
            z = 1j * L(1.3) * np.fft.fft((a.real ** 2 + a.imag ** 2) * a) / N
            z[0] += L(0.5)
            return z

        for _ in range(2):
            k1 = E * F(x)
            k2 = F(E * x + h / 2 * k1)
            k3 = F(E * x + h / 2 * k2)
            k4 = F(E * (E * x + h * k3))
            x = E * (E * x + h / 6 * (k1 + 2 * k2 + 2 * k3)) + h / 6 * k4
        want = np.fft.fftshift(x)
        assert np.linalg.norm(run(kappa) - want) <= 1e-14 * np.linalg.norm(want)
    assert np.isnan(run(-2000.0)).all()
