"""Performance cases of the CME integrator, each one call sequence of a user's program.

A case is one batch (its sizes, precision, integrator and physics) and what the program does
with it per pass:
  * "integrate": give the batch its initial fields (device memory), advance it, take the final
    fields (device memory);
  * "spectrum":  the same, with the power spectra read back to the host after the call, as a
    program does that watches a run;
  * "gradient":  the gradient of the log-spectrum misfit through the whole run (host outputs).

The public API hands every field out in FP64.  A program that chose FP32 has FP32 accuracy and
keeps the results as such, so the FP32 cases end in complex64 / float32.

Parameters follow the repository's workloads (dispersion, pump and detuning ranges, step
sizes).  Runs there take 2000 to 50000 steps per call; a pass here takes fewer steps of the same
call.  Fields start on the continuous-wave state plus noise ("cw", the workloads' start) or on
a developed comb ("comb": a sech envelope over the continuous wave, a run that is continued).
"""
from __future__ import annotations

import math

import numpy as np
import torch


def _case(name, **kw):
    c = dict(kind="integrate", precision="fp32", integrator="rk4ip", D3=0.0, sigma_lo=0.0,
             sigma_hi=8.0, pump_lo=1.5, pump_hi=3.0, kappa=1.0, kappa_ext=0.5, noise=1e-6,
             start="cw", modes=0, kerr=0.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    sweep = dict(sizes="512x256", h=5e-4, D2=0.02, sigma_lo=-2.0, sigma_hi=10.0, pump_lo=2.5,
                 pump_hi=2.5)
    fig1 = dict(sizes="256x4", integrator="strang", h=128 * math.pi / 32768, D2=-0.0125,
                sigma_lo=0.0, sigma_hi=0.0, pump_lo=1.01 * math.sqrt(2.0),
                pump_hi=4.0 * math.sqrt(2.0), kappa=2.0, kappa_ext=1.0, noise=1e-4, modes=201)
    long = dict(h=2e-4, D2=0.01, D3=1e-4)
    return [
        # a program that watches the paper's four-run ensemble: a few steps, then the spectra
        _case("watch_n256_strang_fp32", **dict(fig1, kind="spectrum", steps=8)),
        # one comb of 64 modes in the default precision: nothing but the chain of steps
        _case("single_n64_fp64", sizes="64x1", precision="fp64", steps=200, h=1e-3, D2=0.04,
              sigma_lo=2.5, sigma_hi=2.5, pump_lo=2.0, pump_hi=2.0, noise=1e-4),
        # the paper's ensemble, zero padded 201 in 256, split step, default precision
        _case("fig1_n256_strang_fp64", **dict(fig1, precision="fp64", steps=500)),
        # detuning sweep, one launch of 256 instances: both precisions and both integrators
        _case("sweep_n512_fp32", **dict(sweep, steps=1000)),
        _case("sweep_n512_fp64", **dict(sweep, precision="fp64", steps=100, start="comb")),
        _case("sweep_n512_strang_fp32", **dict(sweep, integrator="strang", steps=2000)),
        # survey of many small combs (an odd number of them), more instances than the GPU holds
        _case("survey_n128_fp32", sizes="128x4099", steps=300, h=1e-3, D2=0.04, start="comb"),
        # instance sizes mixed in one batch
        _case("uneven_n256_4096_fp32", sizes="256x64,1024x64,2048x64,4096x64", steps=500, **long),
        # few wide combs, fewer than the GPU has multiprocessors
        _case("wide_n4096_fp32", sizes="4096x16", steps=500, **long),
        # one octave-spanning comb, wider than one block's memory
        _case("octave_n131072_fp32", sizes="131072x1", steps=200, h=1e-4, D2=2e-4, D3=-4e-7,
              sigma_lo=4.0, sigma_hi=4.0, pump_lo=3.0, pump_hi=3.0, noise=1e-8),
        # fitting a comb to a target spectrum: the supported gradient (FP64), and the FP32 one
        # on fields that FP32 resolves
        _case("gradient_n4096_fp64", kind="gradient", sizes="4096x16", precision="fp64", steps=48,
              start="comb", **long),
        _case("gradient_n1024_fp32", kind="gradient", sizes="1024x32", steps=200, start="comb",
              **dict(long, noise=1e-3, D3=0.0)),
    ]


def draw(rng):
    """One more case of the same ranges; sizes, counts and steps spread over their logarithm."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    precision = rng.choice(["fp32", "fp64"])
    kind = rng.choice(["integrate", "integrate", "integrate", "spectrum", "gradient", "large"])
    integrator = "strang" if kind != "large" and rng.random() < 0.35 else "rk4ip"
    # mode-steps of one pass: below the largest listed case of the precision
    budget = 6e7 if precision == "fp32" else 6e6
    if kind == "gradient":
        budget /= 4
    if kind == "large":
        n = 1 << rng.randint(13, 19)
        count = 1 if n > 65536 else log(1, 4)
        sizes, total, top = "%dx%d" % (n, count), n * count, 200
        D2, D3, h = 2e-4, -4e-7, 1e-4
    else:
        groups = sorted(rng.sample(range(4, 13), rng.choice([1, 1, 1, 2, 3])))
        if kind == "gradient":
            groups = groups[-1:]
        most = 1 if rng.random() < 0.15 else 65536 if precision == "fp64" else 262144
        # about as many modes in each size, an odd number of instances
        share = [(1 << g, max(1, min(2047, log(1, max(2, most // len(groups) >> g))) | 1))
                 for g in groups]
        sizes = ",".join("%dx%d" % s for s in share)
        total, top = sum(n * c for n, c in share), 800
        n = share[-1][0]
        D2, D3 = (0.04, 0.0) if n <= 128 else (0.02, 0.0) if n <= 512 else (0.01, 1e-4)
        h = 1e-3 if n <= 128 else 5e-4 if n <= 512 else 2e-4
    if kind == "gradient":
        top, D3 = 100, 0.0
    steps = max(1, min(top, log(2, max(3, min(top, budget / total)))))
    one = "," not in sizes
    modes = rng.randint(n // 2, n) if one and n >= 16 and rng.random() < 0.25 else 0
    kerr = round(rng.uniform(0.05, 0.3), 3) if integrator == "rk4ip" and kind != "gradient" \
        and rng.random() < 0.15 else 0.0
    start = rng.choice(["cw", "comb"]) if kind != "gradient" else "comb"
    noise = 10.0 ** rng.uniform(-8, -3) if kind != "gradient" else 1e-3
    return _case(None, kind="integrate" if kind == "large" else kind, sizes=sizes,
                 precision=precision, integrator=integrator, steps=steps, h=h, D2=D2, D3=D3,
                 modes=modes, kerr=kerr, start=start, noise=noise)


# ---- inputs (host side, from the seed alone) -----------------------------------------------

def _sizes(case):
    return [tuple(int(v) for v in s.split("x")) for s in case["sizes"].split(",")]


def _cw(sigma, pump, kappa, kappa_ext):
    """Continuous-wave state of the pumped mode: the smallest root of P [(sigma - P)^2 +
    kappa^2/4] = kappa_ext pump^2 (g0 = 1)."""
    r = np.roots([1.0, -2.0 * sigma, sigma * sigma + kappa * kappa / 4, -kappa_ext * pump * pump])
    P = min(x.real for x in r if abs(x.imag) < 1e-9 * max(1.0, abs(x)))
    return math.sqrt(kappa_ext) * pump / (kappa / 2 + 1j * (sigma - P))


def _inputs(case, seed):
    """Per size: (N, sigma [C], pump [C], omega [N], kerr [N] or None, D0 [C, N], target [C, N])."""
    rng = np.random.default_rng(seed)
    out = []
    for N, C in _sizes(case):
        lo, hi = case["sigma_lo"], case["sigma_hi"]
        if (hi - lo, case["pump_hi"] - case["pump_lo"]) == (8.0, 1.5):  # random ensembles
            sigma, pump = rng.uniform(lo, hi, C), rng.uniform(case["pump_lo"], case["pump_hi"], C)
        else:                                                          # sweeps
            sigma, pump = np.linspace(lo, hi, C), np.linspace(case["pump_lo"], case["pump_hi"], C)
        mu = np.arange(N) - N // 2.0
        omega = case["D2"] * mu**2 / 2 + case["D3"] * mu**3 / 6
        kerr = 1.0 + case["kerr"] * mu / (N / 2.0) if case["kerr"] else None
        D0 = rng.standard_normal((C, N, 2)).view(np.complex128)[..., 0] * (case["noise"] / 2**0.5)
        if case["start"] == "comb":
            W = rng.uniform(N / 24.0, N / 8.0, (C, 1))
            D0 += rng.uniform(0.5, 1.5, (C, 1)) / W / np.cosh(np.minimum(np.abs(mu / W), 300.0)) * \
                np.exp(2j * np.pi * rng.uniform(0, 1, (C, 1)) * mu)
        D0[:, N // 2] += [_cw(s, p, case["kappa"], case["kappa_ext"]) for s, p in zip(sigma, pump)]
        if case["modes"]:
            M = case["modes"]
            D0[:, (mu < -(M // 2)) | (mu > M - M // 2 - 1)] = 0.0
        W = rng.uniform(N / 64.0, N / 8.0, (C, 1))
        target = np.log10(rng.uniform(0.01, 1.0, (C, 1)) /
                          np.cosh(np.minimum(np.abs(mu / W), 300.0))**2 + 1e-20)
        out.append((N, sigma, pump, omega, kerr, D0, target))
    return out


# ---- a pass ---------------------------------------------------------------------------------

_stream = None


def _program_stream():
    """The one stream that the program works on: its batches run one after the other."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    from paper_1307_3428_gb300 import cme

    insts, fields, targets = [], [], []
    for N, sigma, pump, omega, kerr, D0, target in _inputs(case, seed):
        kappa = np.full(N, case["kappa"])
        insts += [cme.Instance(N, kappa, omega, 1.0, case["kappa_ext"], pump[i], sigma[i],
                               np.zeros(N, complex), case["modes"] or None, kerr)
                  for i in range(len(sigma))]
        fields.append(D0.reshape(-1))
        targets.append(target.reshape(-1))
    stream = _program_stream()
    single = case["precision"] == "fp32"
    batch = cme.Batch(insts, precision=cme.FP32 if single else cme.FP64,
                      integrator=cme.STRANG if case["integrator"] == "strang" else cme.RK4IP,
                      use_graph=case["kind"] == "integrate", stream=stream.cuda_stream)
    D0 = torch.from_numpy(np.concatenate(fields)).cuda()
    out = torch.empty_like(D0)
    torch.cuda.synchronize()
    return dict(case=case, batch=batch, stream=stream, D0=D0, out=out,
                out32=torch.empty(D0.shape, dtype=torch.complex64, device="cuda"),
                target=np.concatenate(targets), power=cme.POWER, single=single)


def run(state):
    c, b = state["case"], state["batch"]
    b.set_state_device(state["D0"].data_ptr())
    if c["kind"] == "gradient":
        g = b.grad(c["h"], c["steps"], state["target"])
        if state["single"]:
            g = {k: v.astype(np.complex64 if v.dtype.kind == "c" else np.float32)
                 for k, v in g.items()}
        return g
    b.step(c["h"], c["steps"])
    if c["kind"] == "spectrum":
        power = b.spectrum(state["power"])
        return power.astype(np.float32) if state["single"] else power
    b.get_state_device(state["out"].data_ptr())
    if not state["single"]:
        return state["out"]
    with torch.cuda.stream(state["stream"]):
        state["out32"].copy_(state["out"])
    return state["out32"]


def work(case):
    """Transforms at 5 N log2 N, plus the pointwise work, per mode-step; the fields in and out.

    A gradient's backward step holds as many transforms as its forward step."""
    modes = sum(n * c for n, c in _sizes(case))
    per = (40, 80) if case["integrator"] == "rk4ip" else (10, 40)
    flops = sum(n * c * (per[0] * math.log2(n) + per[1]) for n, c in _sizes(case)) * case["steps"]
    io = 16 if case["kind"] == "spectrum" else 32
    if case["kind"] == "gradient":
        flops, io = 2 * flops, 64
    return {"bytes": float(modes * (io + 24)), "flops": float(flops)}


# ---- the same in plain torch, 64 bits --------------------------------------------------------

def _integrate(case, N, L, g, pump, D, keep):
    """`steps` steps of D [C, N] (transform order); the textbook forms of both integrators."""
    h = case["h"]
    E = torch.exp(L * (h / 2))
    if case["integrator"] == "strang":
        half = torch.zeros_like(L)
        half[:, :1] = torch.where(L[:, :1] == 0, h / 2 + 0j, (E[:, :1] - 1) /
                                  torch.where(L[:, :1] == 0, 1 + 0j, L[:, :1])) * pump
        for _ in range(case["steps"]):
            D = E * D + half
            a = torch.fft.ifft(D) * N
            D = torch.fft.fft(a * torch.exp(1j * h * (a.real**2 + a.imag**2))) / N * keep
            D = E * D + half
        return D
    first = torch.zeros(N, dtype=torch.complex128, device=D.device)
    first[0] = 1.0

    def F(x):
        a = torch.fft.ifft(x) * N
        return 1j * g * torch.fft.fft((a.real**2 + a.imag**2) * a) / N * keep + pump * first

    for _ in range(case["steps"]):
        Ia = E * D
        k1 = E * F(D)
        k2 = F(Ia + (h / 2) * k1)
        k3 = F(Ia + (h / 2) * k2)
        k4 = F(E * (Ia + h * k3))
        D = E * (Ia + (h / 6) * (k1 + 2 * k2 + 2 * k3)) + (h / 6) * k4
    return D


def exact(case, seed):
    fields, grads = [], []
    for N, sigma, pump, omega, kerr, D0, target in _inputs(case, seed):
        roll = torch.fft.ifftshift

        def dev(v):
            return torch.from_numpy(np.ascontiguousarray(v)).cuda()

        mu = np.arange(N) - N // 2
        M = case["modes"] or N
        keep = roll(dev(((mu >= -(M // 2)) & (mu <= M - M // 2 - 1)).astype(float)))
        g = 1.0 if kerr is None else roll(dev(kerr))
        w, kappa = roll(dev(omega)), torch.full((N,), float(case["kappa"]), device="cuda",
                                                dtype=torch.float64)
        sig, p, D = dev(sigma), dev(pump + 0j), roll(dev(D0), dim=-1)
        want = case["kind"] == "gradient"
        C = len(sigma)
        if want:
            w, kappa = w.repeat(C, 1), kappa.repeat(C, 1)
        leaves = [w, kappa, sig, p, D]
        for v in leaves:
            v.requires_grad_(want)
        with torch.set_grad_enabled(want):
            L = torch.complex((-kappa / 2).expand(C, N), w - w[..., :1] - sig[:, None])
            s = math.sqrt(case["kappa_ext"]) * p[:, None]
            E = _integrate(case, N, L, g, s, D, keep)
            if want:
                T = roll(dev(target), dim=-1)
                loss = ((torch.log10(E.real**2 + E.imag**2 + 1e-20) - T)**2).sum(dim=-1)
                dw, dk, ds, dp, dD = torch.autograd.grad(loss.sum(), leaves)
        if want:
            m = roll(dev(mu.astype(float)))
            back = lambda v: torch.fft.fftshift(v, dim=-1).reshape(-1).cpu().numpy()  # noqa: E731
            grads.append({"loss": loss.detach().cpu().numpy(), "d_sigma": ds.cpu().numpy(),
                          "d_A_in": dp.cpu().numpy(), "d_D2": (dw * m**2 / 2).sum(-1).cpu().numpy(),
                          "d_D3": (dw * m**3 / 6).sum(-1).cpu().numpy(), "d_omega": back(dw),
                          "d_kappa": back(dk), "d_D0": back(dD)})
        else:
            fields.append(torch.fft.fftshift(E, dim=-1).reshape(-1))
    if grads:
        return {k: np.concatenate([v[k] for v in grads]) for k in grads[0]}
    D = torch.cat(fields)
    return (D.real**2 + D.imag**2).cpu().numpy() if case["kind"] == "spectrum" else D
