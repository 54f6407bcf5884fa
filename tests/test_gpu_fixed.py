"""FP64 transforms and right-hand side (computed in 64-bit fixed point, csrc/cme_fixed.cuh) against
extended precision: unrelated modes, a comb on a continuous wave, a wave packet of one sample,
modes of very different size, and magnitudes near both ends of the FP64 range.

Bounds.  An FP64 transform rounds every value once per level: relative 2-norm error of about
2^-53 per level.  The Kerr term triples the relative error of the time samples, and the samples
that carry it are at most a factor of about 2 above the 2-norm's share (the fields below), so the
right-hand side gets 4 x (levels + 2) roundings."""
import numpy as np
import pytest

from paper_1307_3428_gb300 import cme

pytestmark = pytest.mark.gpu
L = np.clongdouble
ULP = 2.0 ** -53


def fields(N):
    rng = np.random.default_rng(1307 + N)
    mu = np.arange(N) - N // 2
    r = rng.standard_normal((N, 2)).view(complex)[:, 0]
    comb = 1e-9 * r + 0.3 / np.cosh(mu / (N / 16)) * np.exp(2j * np.pi * 0.3 * mu)
    comb[N // 2] += 0.5
    cw = 1e-6 * r
    cw[N // 2] += 1.2 + 0.4j
    return {"random": r / np.sqrt(N), "comb": comb, "cw": cw,
            "mixed": r * 10.0 ** rng.uniform(-12, 0, N)}


def batch(D, **kw):
    N = D.size
    return cme.Batch([cme.Instance(N, np.ones(N), np.zeros(N), 1.3, 0.5, 0.7, 1.0, D)], **kw)


def rel(x, y):
    return float(np.linalg.norm(x - y) / np.linalg.norm(y))


SHAPES = [(4, 4), (8, 8), (16, 8), (16, 16), (32, 8), (64, 2), (64, 4), (64, 8), (64, 16),
          (128, 2), (128, 8), (256, 4), (256, 8), (512, 4), (512, 8), (1024, 8), (2048, 8),
          (2048, 16), (4096, 8), (4096, 16)]


@pytest.mark.parametrize("N,R", SHAPES)
def test_transforms_and_rhs_against_extended_precision(N, R):
    levels = int(np.log2(N))
    for name, D in fields(N).items():
        b = batch(D, radix=R)
        x = np.fft.ifftshift(D.astype(L))
        a = np.fft.ifft(x) * N
        assert rel(b.transform(1), a) <= ULP * (levels + 2), name
        assert rel(b.transform(-1), np.fft.fft(x)) <= ULP * (levels + 2), name
        y = np.fft.fft((a.real ** 2 + a.imag ** 2) * a) / N * (1j * L(1.3))
        y[0] += np.sqrt(L(0.5)) * L(0.7)
        assert rel(b.eval_rhs(), np.fft.fftshift(y)) <= ULP * 4 * (levels + 2), name
        b.close()


@pytest.mark.parametrize("N", [16, 64, 512, 4096])
@pytest.mark.parametrize("scale", [1e-300, 1e-160, 1e150, 1e300])
def test_transform_near_the_ends_of_the_fp64_range(N, scale):
    D = fields(N)["random"] * scale
    b = batch(D)
    x = np.fft.ifftshift((D / scale).astype(L))
    got = b.transform(1).astype(L) / L(scale)
    # the scaled input itself is rounded once
    assert rel(got, np.fft.ifft(x) * N) <= ULP * (np.log2(N) + 4)


@pytest.mark.parametrize("N", [16, 512])
def test_groups_of_one_block_scale_apart(N):
    """Instances that share a warp or a block keep their own scale: each result has the bits it
    has alone, whatever its neighbours' magnitude."""
    D = [fields(N)["random"] * s for s in (1.0, 1e-200, 1e100, 0.0, 1e-310, 1e-9)]
    insts = [cme.Instance(N, np.ones(N), np.zeros(N), 1.3, 0.5, 0.7, 1.0, d) for d in D]
    for call in (lambda b: b.transform(1), lambda b: b.eval_rhs()):
        together = call(cme.Batch(insts, radix=8)).reshape(len(D), N)
        for i, inst in enumerate(insts):
            np.testing.assert_array_equal(together[i], call(cme.Batch([inst], radix=8)))


@pytest.mark.parametrize("N", [16, 64, 512, 4096])
def test_zero_modes_stay_zero(N):
    """A continuous wave has no four-wave mixing into other modes: they are zero, not a rounding
    unit."""
    D = np.zeros(N, complex)
    b = batch(D)
    b.step(1e-3, 3)
    got = b.get_state()
    assert got[N // 2] != 0
    got[N // 2] = 0
    assert not got.any()


@pytest.mark.parametrize("N", [16, 512, 4096])
@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e200])
def test_non_finite_fields_are_reported(N, bad):
    D = fields(N)["comb"]
    b = batch(D)
    D[1] = bad
    b.set_state(D)
    b.step(1e-3, 3)
    assert b.status()[0] == 1


def strang_extended(D, h, n, sigma=1.0, g0=1.3, pump=np.sqrt(L(0.5)) * L(0.7)):
    """n Strang steps in extended precision (kappa = 1, omega = 0)."""
    N = D.size
    Lm = L(-0.5) - 1j * L(sigma)
    half = np.exp(Lm * L(h) / 2)
    x = np.fft.ifftshift(D.astype(L))
    for _ in range(n):
        x = half * x
        x[0] += (half - 1) / Lm * pump
        a = np.fft.ifft(x) * N
        x = np.fft.fft(a * np.exp(1j * L(g0) * L(h) * (a.real ** 2 + a.imag ** 2))) / N
        x = half * x
        x[0] += (half - 1) / Lm * pump
    return np.fft.fftshift(x)


@pytest.mark.parametrize("N,R", [(4, 4), (16, 16), (64, 2), (64, 4), (256, 4), (512, 8), (4096, 8)])
@pytest.mark.parametrize("phase", [1e-9, 1e-4, 0.03, 0.2, 0.45, 0.97, 1.1, 7.0])
def test_split_step_phases(N, R, phase):
    """Kerr phases from far below to above the Taylor series' range (1), on fields whose largest
    sample has that phase.  Per step the linear flows round each mode three times and the Kerr
    flow is one right-hand side."""
    h = 1e-2
    for name, D in fields(N).items():
        a = np.fft.ifft(np.fft.ifftshift(D)) * N
        D = D * np.sqrt(phase / (1.3 * h)) / np.abs(a).max()
        b = batch(D, radix=R, integrator=cme.STRANG)
        b.step(h, 2)
        assert rel(b.get_state(), strang_extended(D, h, 2)) <= ULP * 8 * (np.log2(N) + 4), name
        b.close()


def test_split_step_phases_of_one_block_scale_apart():
    D = [fields(64)["random"] * s for s in (1.0, 1e-3, 30.0, 1e-200, 0.0)]
    insts = [cme.Instance(64, np.ones(64), np.zeros(64), 1.3, 0.5, 0.7, 1.0, d) for d in D]
    kw = dict(radix=8, integrator=cme.STRANG)
    b = cme.Batch(insts, **kw)
    b.step(1e-2, 3)
    together = b.get_state().reshape(len(D), 64)
    for i, inst in enumerate(insts):
        one = cme.Batch([inst], **kw)
        one.step(1e-2, 3)
        np.testing.assert_array_equal(together[i], one.get_state())


def test_fp64_plan_by_group_size():
    """Values per thread of FP64 groups: 2 (N <= 128) and 4 (N <= 512) while their warps are at most
    two per scheduler, then more; one block per instance at N = 2048; 2 values only on request at
    N = 64 and 128."""
    torch = pytest.importorskip("torch")
    room = 8 * torch.cuda.get_device_properties(0).multi_processor_count   # warps
    inst = {N: cme.Instance(N, np.ones(N), np.zeros(N), 1.0, 0.5, 0.7, 1.0, np.zeros(N, complex))
            for N in (16, 32, 64, 128, 256, 512, 1024, 2048)}
    for N, count, radix in ((16, 1, 2), (16, 4 * room, 2), (16, 4 * room + 1, 8), (32, 2 * room, 2),
                            (64, room, 2), (64, room + 1, 4), (128, room // 2, 2),
                            (128, room // 2 + 1, 4), (128, room + 1, 8), (256, room // 2, 4),
                            (256, room // 2 + 1, 8), (512, room // 4, 4), (512, room // 4 + 1, 8),
                            (1024, 1, 8), (2048, 1, 8)):
        b = cme.Batch([inst[N]] * count)
        assert (b.plan(0)["radix"], b.plan(0)["cluster"]) == (radix, 1), (N, count, b.plan(0))
        b.close()
    with pytest.raises(cme.CmeError):
        cme.Batch([inst[16]], radix=2)
