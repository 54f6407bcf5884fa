"""The FP64 steps' 64-bit fixed point (csrc/cme_fixed.cuh) on the CPU: the device source itself, built
for the host with overflow checks on every signed sum, product and shift, for every compiled launch
shape, against extended precision.

The fields are those that reach a bound: a spectrum of equal modes is one sample in time, the
largest sample that a transform can leave, and a sech spectrum is a pulse; sixteen mantissas over
one octave move the largest value from just above a power of two to just below the next.

Bounds: an FP64 transform rounds every value once per level, a relative 2-norm error of 2^-53
per level.  The Kerr term triples the relative error of the samples, and in these fields the samples
that carry the term carry the 2-norm too; so the right-hand side gets 4 x (levels + 2) roundings.  A
step adds one right-hand side (the split step's Kerr flow, the weighted sum of the four stages) and
rounds each mode a few times: 8 x (levels + 4), as in test_gpu_fixed.py."""
import concurrent.futures as cf
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1307_3428_gb300", "csrc")
L = np.clongdouble
ULP = 2.0 ** -53
G0, KAPPA, SIGMA = 1.3, 1.0, 1.0

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")


def shapes():
    text = open(os.path.join(CSRC, "cme_launch.cuh")).read()
    macro = re.search(r"#define CME_FOR_EACH_SHAPE\(X\)(.*?[^\\])\n", text, re.S).group(1)
    return [(int(a), int(b)) for a, b in re.findall(r"X\((\d+), (\d+)\)", macro)]


def host_build(out, logN, R):
    exe = str(out / f"fixed_{logN}_{R}")
    subprocess.run(["g++", "-std=c++17", "-O1", "-g1", "-ffp-contract=off",
                    "-fsanitize=signed-integer-overflow,shift", "-fno-sanitize-recover=all",
                    "-I", os.path.join(ROOT, "tests", "host_fixed"), "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), f"-DCASE_LOGN={logN}", f"-DCASE_R={R}",
                    os.path.join(ROOT, "tests", "host_fixed", "fixed.cpp"), "-o", exe],
                   check=True, capture_output=True)
    return exe


@pytest.fixture(scope="module")
def builds(tmp_path_factory):
    out = tmp_path_factory.mktemp("fixed")
    with cf.ThreadPoolExecutor(os.cpu_count()) as pool:
        made = pool.map(lambda s: host_build(out, *s), shapes())
        return dict(zip(shapes(), made))


def run(exe, what, fields, tmp_path, g0=G0, pump=0.0, h=1e-3, steps=1):
    """`fields` [n, N] (transform order) after the right-hand side or `steps` steps."""
    src, dst = tmp_path / "in", tmp_path / "out"
    np.ascontiguousarray(fields, complex).tofile(src)
    r = subprocess.run([exe, what, *(repr(float(v)) for v in (g0, KAPPA, pump, h)), str(steps), src, dst],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[:400]
    return np.fromfile(dst, complex).reshape(fields.shape)


def pulses(N):
    """Spectra of short pulses: equal modes (real, imaginary, at 45 degrees, at a time between two
    samples) and sech envelopes of widths N/16 to N, each at 16 sizes in [1/2, 1)."""
    mu = np.fft.ifftshift(np.arange(N) - N // 2)
    out = [np.ones(N), 1j * np.ones(N), (1 + 1j) * np.ones(N), np.exp(2j * np.pi * 0.3 * mu)]
    out += [1 / np.cosh(mu / (N / w)) for w in (16, 8, 4, 2, 1)]
    size = 2.0 ** (np.arange(-16, 0) / 16)
    return (size[:, None, None] * np.array(out)).reshape(-1, N)


def rel(x, y):
    return np.linalg.norm(x - y, axis=-1) / np.linalg.norm(y, axis=-1)


def rhs_extended(D, g0=G0):
    a = np.fft.ifft(D.astype(L)) * D.shape[-1]
    return 1j * L(g0) * np.fft.fft((a.real ** 2 + a.imag ** 2) * a) / D.shape[-1]


@pytest.mark.parametrize("logN,R", shapes())
def test_kerr_term_of_short_pulses(builds, tmp_path, logN, R):
    D = pulses(1 << logN)
    err = rel(run(builds[logN, R], "rhs", D, tmp_path), rhs_extended(D))
    assert err.max() <= ULP * 4 * (logN + 2), (int(err.argmax()), float(err.max()))


def propagator(D, t):
    return np.exp((L(-KAPPA / 2) - 1j * L(SIGMA)) * L(t))


def rk4ip_extended(D, h, pump):
    D, h, E = D.astype(L), np.longdouble(h), propagator(D, np.longdouble(h) / 2)

    def F(x):
        y = rhs_extended(x)
        y[..., 0] += L(pump)
        return y

    k1 = E * F(D)
    k2 = F(E * D + h / 2 * k1)
    k3 = F(E * D + h / 2 * k2)
    k4 = F(E * (E * D + h * k3))
    return E * (E * D + h / 6 * (k1 + 2 * k2 + 2 * k3)) + h / 6 * k4


def strang_extended(D, h, pump):
    D, E = D.astype(L), propagator(D, np.longdouble(h) / 2)
    into = (E - 1) / (L(-KAPPA / 2) - 1j * L(SIGMA)) * L(pump)
    D = E * D
    D[..., 0] += into
    a = np.fft.ifft(D) * D.shape[-1]
    D = E * np.fft.fft(a * np.exp(1j * L(G0) * L(h) * (a.real ** 2 + a.imag ** 2))) / D.shape[-1]
    D[..., 0] += into
    return D


@pytest.mark.parametrize("logN,R", shapes())
@pytest.mark.parametrize("what,step,phase", [("rk4ip", rk4ip_extended, 0.2),
                                             ("strang", strang_extended, 0.2),
                                             ("strang", strang_extended, 5.0)])
def test_steps_of_short_pulses(builds, tmp_path, logN, R, what, step, phase):
    """phase: the Kerr phase of the largest sample of each shape's sixteen sizes (the split step's
    series ends at 1)."""
    N = 1 << logN
    for D in np.moveaxis(pulses(N).reshape(16, -1, N), 1, 0):
        h = phase / (G0 * np.abs(np.fft.ifft(D) * N).max() ** 2)
        err = rel(run(builds[logN, R], what, D, tmp_path, pump=0.5, h=h), step(D, h, 0.5))
        assert err.max() <= ULP * 8 * (logN + 4), (int(err.argmax()), float(err.max()))


@pytest.mark.parametrize("logN,R", shapes())
@pytest.mark.parametrize("what", ["rk4ip", "strang"])
def test_overflowing_fields_become_nan(builds, tmp_path, logN, R, what):
    """A field whose |a|^2 leaves the FP64 range has no result: every mode is NaN or infinite after
    the step, and instances in the same block keep the bits they have alone."""
    N = 1 << logN
    rng = np.random.default_rng(5)
    D = np.tile(rng.standard_normal((N, 2)).view(complex)[:, 0], (4, 1))
    D[1] *= 1e200
    D[3, 1] = 1e155
    got = run(builds[logN, R], what, D, tmp_path, pump=0.5)
    assert not np.isfinite(got[[1, 3]]).any()
    alone = run(builds[logN, R], what, D[:1], tmp_path, pump=0.5)
    np.testing.assert_array_equal(got[[0, 2]], np.concatenate([alone, alone]))


@pytest.mark.parametrize("logN,R", shapes())
def test_unpumped_zero_field_stays_zero(builds, tmp_path, logN, R):
    D = np.zeros((3, 1 << logN), complex)
    assert not run(builds[logN, R], "rk4ip", D, tmp_path, steps=3).any()
    D[1, 1] = 1e-160           # its Kerr term lies far below the range: no mixing into mode 0
    got = run(builds[logN, R], "rk4ip", D, tmp_path, steps=3)
    assert got[1, 1] != 0 and not np.delete(got[1], 1).any() and not got[[0, 2]].any()


@pytest.mark.parametrize("pump", [1e-300, 3e-308, 1e-310])
def test_smallest_pumps(builds, tmp_path, pump):
    """A pump near the end of the range (its half step subnormal) on a zero field: h pump after a
    short step, to the spacing of the range's end."""
    h = 1e-3
    for logN, R in ((4, 2), (6, 8), (9, 4)):
        got = run(builds[logN, R], "rk4ip", np.zeros((1, 1 << logN), complex), tmp_path, pump=pump,
                  h=h)[0]
        assert abs(got[0] - pump * h) <= 2e-3 * pump * h + 8 * 2.0 ** -1074
        assert not got[1:].any()


def combs(N, rng, n):
    """Sech envelopes of a random time and width on a continuous wave and noise."""
    mu = np.fft.ifftshift(np.arange(N) - N // 2)
    W = rng.uniform(N / 24, N / 8, (n, 1))
    D = rng.standard_normal((n, N, 2)).view(complex)[..., 0] * 10.0 ** rng.uniform(-8, -6, (n, 1))
    D += (rng.uniform(0.5, 1.5, (n, 1)) / W / np.cosh(np.minimum(np.abs(mu / W), 300)) *
          np.exp(2j * np.pi * rng.uniform(0, 1, (n, 1)) * mu))
    D[:, 0] += rng.uniform(0.3, 1.5, n) * np.exp(2j * np.pi * rng.uniform(0, 1, n))
    return D


def small_mode_errors(D, got, h, pump):
    """Root mean square error over the modes below 1e-4, of `got` and of FP64 arithmetic."""
    want = rk4ip_extended(D, h, pump)
    E, e1, e2 = (propagator(D, np.longdouble(h) / 2), propagator(D, np.longdouble(h) / 2) - 1,
                 propagator(D, h) - 1)
    E, e1, e2, N = complex(E), complex(e1), complex(e2), D.shape[-1]

    def F(x):
        a = np.fft.ifft(x) * N
        y = 1j * G0 * (np.fft.fft((a.real ** 2 + a.imag ** 2) * a) / N)
        y[..., 0] += pump
        return y

    k1 = E * F(D)
    k2 = F(D + (e1 * D + h / 2 * k1))
    k3 = F(D + (e1 * D + h / 2 * k2))
    k4 = F(D + (e2 * D + h * E * k3))
    plain = D + (e2 * D + h / 6 * (E * (k1 + 2 * k2 + 2 * k3) + k4))
    small = np.abs(D) < 1e-4
    return [float(np.sqrt(np.mean(np.abs((x - want)[small]) ** 2))) for x in (got, plain)]


@pytest.mark.parametrize("logN,R", [s for s in shapes() if s[0] >= 4])
def test_small_modes_of_an_rk4ip_step(builds, tmp_path, logN, R):
    """One scale per instance leaves modes far below the pumped one fewer bits than FP64 numbers
    have.  What counts is the error of a step on them: at most twice that of FP64 arithmetic with
    numpy's transforms."""
    N = 1 << logN
    D = combs(N, np.random.default_rng(logN), 128 if N < 1024 else 32)
    h = 1e-3 if N <= 128 else 5e-4 if N <= 512 else 2e-4
    fixed, plain = small_mode_errors(D, run(builds[logN, R], "rk4ip", D, tmp_path, pump=1.5, h=h),
                                     h, 1.5)
    assert fixed <= 2 * plain


@pytest.mark.parametrize("logN,R", [(9, 4), (9, 8), (12, 8)])
def test_increment_unit(builds, tmp_path, logN, R):
    """A continuous wave of 1.3 with modes of 1e-6, h = 2e-4: the increment, about 1e-3, is held to
    2^-60 of itself, so the small modes end within 2e-21 (FP64 instructions: 1.6e-21 to 4.9e-21)."""
    rng = np.random.default_rng(1)
    D = 1e-6 * rng.standard_normal((16, 1 << logN, 2)).view(complex)[..., 0]
    D[:, 0] += 1.2 + 0.4j
    got = run(builds[logN, R], "rk4ip", D, tmp_path, pump=0.5, h=2e-4)
    assert small_mode_errors(D, got, 2e-4, 0.5)[0] <= 2e-21


@pytest.mark.parametrize("logN,R", [s for s in shapes() if s[0] >= 4 and s[1] > 2])
def test_output_0_has_no_bias(builds, tmp_path, logN, R):
    """Output 0 sums the products with twiddle 1, whose floors are corrected by their mean.  Two strong
    modes on noise, all modes with sum 0: what a transform returns there is its error, and its mean
    over the fields has to stay below one field's rounding noise."""
    N, n = 1 << logN, 256
    x = np.random.default_rng(N).standard_normal((n, N, 2)).view(complex)[..., 0]
    x[:, 0] *= 1e6
    x[:, 3] = 0
    x[:, 3] = -x.astype(L).sum(axis=1)
    err = (run(builds[logN, R], "idft", x, tmp_path)[:, 0] - x.astype(L).sum(axis=1)).astype(complex)
    for e in (err.real, err.imag):
        assert abs(e.mean()) <= e.std()
