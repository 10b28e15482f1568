"""Performance cases of the diffractive-storage engine: what its users have it do.

A user designs a stack of K thickness layers for N_w wavelength channels and has
the engine evaluate it through ``DiffractiveStack`` (or ``DosFunction`` under
autograd):

* ``step``      one design step, forward + objective + adjoint, as the
                fine-tuning driver calls it (``DiffractiveStack.step``);
* ``autograd``  the same gradient through ``DosFunction`` and a torch objective;
* ``vaccinate`` a design step with freshly displaced layers (forward, loss,
                backward as three calls, since the displacement changes each time);
* ``evaluate``  scoring of a finished design at a phase bit depth: quantise the
                thickness, forward without checkpoints, PSNR, efficiency;
* ``propagate`` one free-space gap and its adjoint on caller fields.

``listed()`` gives the sizes that stand for these uses, ``draw`` more of the same
ranges.  ``exact`` restates the method in 64-bit torch operations.
"""
import math

import numpy as np
import torch

from paper_2604_02624_gb300.api import DiffractiveStack, DosFunction, quantize_thickness

NM = 1e-9


def _case(name, kind, n, m, layers, channels, fov, lo=450.0, hi=750.0, gap=210.0, kappa=0.01,
          path="auto", loss="mse", evanescent="decay", bin=1, bits=6, medium=1.0, base=0.0, unequal=False):
    return dict(name=name, kind=kind, n=n, m=m, layers=layers, channels=channels, fov=fov, lo=lo, hi=hi,
                gap=gap, kappa=kappa, path=path, loss=loss, evanescent=evanescent, bin=bin, bits=bits,
                medium=medium, base=base, unequal=unequal)


def listed():
    return [
        # the smallest design: one layer, four wavelengths; a fine-tuning iteration is all launches and latency
        _case("step_4x64", "step", 64, 128, 1, 4, 32, 500, 740, 40, 0.0),
        # the six-wavelength, two-layer experiment, trained under torch autograd
        _case("autograd_6x200", "autograd", 200, 400, 2, 6, 50, 500, 740, 100),
        # an ordinary five-layer design: 256 wavelengths fit one step of a desk-side training run
        _case("step_256x200", "step", 200, 400, 5, 256, 50, kappa=0.0),
        # the same design vaccinated against misalignment: every step has its own layer displacements
        _case("vaccinate_256x200", "vaccinate", 200, 400, 5, 256, 50),
        # the flagship: thousands of channels, five layers
        _case("step_4096x200", "step", 200, 400, 5, 4096, 50),
        # the high-precision design: eight larger layers
        _case("step_2048x256", "step", 256, 512, 8, 2048, 64, gap=160),
        # scoring a finished design (PSNR and efficiency of every channel) at 6 bits of phase depth
        _case("evaluate_1024x200", "evaluate", 200, 400, 5, 1024, 50),
        # one gap on caller fields, both directions: beam analysis beside the design loop
        _case("propagate_64x256", "propagate", 256, 512, 1, 64, 64, gap=160),
        # odd and ragged sizes: odd layer, unequal gaps, a dense medium, a base thickness, the scaled loss
        _case("step_96x101", "step", 101, 256, 3, 96, 41, gap=55, loss="mse_scaled", evanescent="zero",
              medium=1.33, base=120.0, unequal=True),
        # many channels of a small layer, scored on integrating detector pixels
        _case("step_2048x64", "step", 64, 128, 3, 2048, 32, gap=60, bin=4),
        # the tensor-core form of the transforms, two bf16 parts, on the high-precision geometry
        _case("gemm_128x256", "autograd", 256, 512, 8, 128, 64, gap=160, path="dft_gemm"),
        # the three-part form on the experiment's geometry
        _case("gemm3_24x200", "autograd", 200, 400, 2, 24, 50, gap=100, path="dft_gemm_x3"),
    ]


def _cost(c):
    return c["channels"] * (c["layers"] + 1) * c["m"] ** 2 * (8.0 if c["path"].startswith("dft_gemm") else 1.0)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "autograd", "vaccinate", "evaluate", "propagate"])
    m = rng.choice([64, 128, 200, 256, 400, 400, 400, 512, 512])
    # mostly zero-padded to at least twice the layer, now and then less
    n = rng.randint(max(9, m // 4), m // 2) if rng.random() < 0.85 else rng.randint(m // 2, (3 * m) // 4)
    if rng.random() < 0.4 and n > m // 4:
        n = m // 2
    fov = rng.randint(max(3, n // 6), n // 2)
    fov -= (n - fov) % 2
    divisors = [b for b in (2, 3, 4, 5) if fov % b == 0]
    path = "auto"
    if kind in ("step", "autograd", "evaluate") and rng.random() < 0.15:
        path = rng.choice(["dft_gemm", "dft_gemm_x3"])
    layers = 1 if kind == "propagate" else rng.randint(1, 8)
    most = 0.4e9 / ((layers + 1) * m * m * (8.0 if path != "auto" else 1.0))
    channels = int(round(math.exp(rng.uniform(math.log(1.0), math.log(max(2.0, min(4096.0, most)))))))
    lo = rng.uniform(430.0, 520.0)
    return dict(kind=kind, n=n, m=m, layers=layers, channels=max(1, channels), fov=fov, lo=lo,
                hi=lo + rng.uniform(60.0, 300.0), gap=round(rng.uniform(30.0, 210.0), 1),
                kappa=rng.choice([0.0, 0.01]), path=path, loss=rng.choice(["mse", "mse_scaled"]),
                evanescent=rng.choice(["decay", "decay", "zero"]),
                bin=rng.choice(divisors) if divisors and kind == "step" and rng.random() < 0.3 else 1,
                bits=rng.choice([1, 4, 6, 8]), medium=rng.choice([1.0, 1.0, 1.33]),
                base=rng.choice([0.0, 120.0]), unequal=rng.random() < 0.3)


# ------------------------------------------------------------------ the design and its inputs
def _design(c):
    lam = np.linspace(c["lo"], c["hi"], c["channels"]) * NM
    lam_m = 0.5 * (c["lo"] + c["hi"]) * NM
    gaps = np.full(c["layers"] + 1, c["gap"] * lam_m)
    if c["unequal"]:
        gaps *= 1.0 + 0.25 * np.arange(c["layers"] + 1)
    n_index = 1.7 + 0.02 * (lam_m - lam) / lam_m if c["unequal"] else np.full(lam.shape, 1.7)
    return dict(lam=lam, lam_m=lam_m, gaps=gaps, n_index=n_index, pitch=0.5 * lam_m)


def _targets(gen, channels, fov, dev):
    """Grey low-resolution images, box-smoothed over in-bounds neighbours, brought to fov x fov."""
    src = min(28, fov)
    low = torch.rand((channels, 1, src, src), generator=gen, device=dev)
    low = torch.nn.functional.avg_pool2d(low, 3, stride=1, padding=1, count_include_pad=False)
    return torch.nn.functional.interpolate(low, size=(fov, fov), mode="nearest")[:, 0].contiguous()


def _inputs(c, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    d = _design(c)
    if c["kind"] == "propagate":
        f = torch.randn((c["channels"], c["n"], c["n"], 2), generator=gen, device=dev)
        return dict(field=torch.view_as_complex(f))
    h = torch.rand((c["layers"], c["n"], c["n"]), generator=gen, device=dev) * float(d["lam_m"])
    out = dict(h=h, T=_targets(gen, c["channels"], c["fov"] // c["bin"], dev))
    if c["kind"] == "vaccinate":
        # lateral displacements of up to a few features, axial ones of a wavelength
        r = torch.rand((c["layers"], 3), generator=gen, device=dev).cpu().numpy().astype(np.float64) * 2.0 - 1.0
        out["shift"] = r * np.array([3.0 * d["pitch"], 3.0 * d["pitch"], d["lam_m"]])
    return out


def prepare(case, seed):
    d, s = _design(case), _inputs(case, seed)
    s["case"] = case
    s["h_max"] = float(d["lam_m"])
    s["stack"] = DiffractiveStack(
        n=case["n"], m=case["m"], n_layers=case["layers"], lambdas=d["lam"], gaps=d["gaps"], pitch=d["pitch"],
        n_index=d["n_index"], kappa=case["kappa"], fov=case["fov"], n_medium=case["medium"],
        h_base=case["base"] * NM, evanescent=case["evanescent"], loss=case["loss"], path=case["path"],
        detector_bin=case["bin"])
    if case["kind"] == "autograd":
        s["h"].requires_grad_(True)
    if case["kind"] == "step":
        dev, k = s["h"].device, (case["channels"], case["fov"], case["fov"])
        s["grad"] = torch.empty_like(s["h"])
        s["I"] = torch.empty(k, device=dev)
        s["psnr"] = torch.empty(case["channels"], device=dev)
    return s


def run(state):
    kind, stack = state["case"]["kind"], state["stack"]
    if kind == "step":
        stack.step(state["h"], state["T"], grad_out=state["grad"], intensity_out=state["I"], psnr_out=state["psnr"])
        return dict(grad=state["grad"], I=state["I"], psnr=state["psnr"])
    if kind == "autograd":
        I = DosFunction.apply(state["h"], stack)
        T = state["T"]
        if state["case"]["loss"] == "mse_scaled":
            sigma = ((I * T).sum((1, 2)) / (I * I).sum((1, 2))).detach()
            loss = ((sigma[:, None, None] * I - T) ** 2).mean()
        else:
            loss = ((I - T) ** 2).mean()
        grad, = torch.autograd.grad(loss, state["h"])
        return dict(grad=grad, I=I.detach(), loss=loss.detach())
    if kind == "vaccinate":
        stack.set_misalignment(state["shift"])
        I = stack.forward(state["h"])
        _, psnr, dLdI = stack.loss(state["T"], read=False)
        return dict(grad=stack.backward(dLdI), I=I, psnr=psnr)
    if kind == "evaluate":
        hq = quantize_thickness(state["h"], state["h_max"], state["case"]["bits"])
        I = stack.forward(hq, save_for_backward=False)
        _, psnr, _ = stack.loss(state["T"], read=False, grad=False)
        return dict(I=I, psnr=psnr, efficiency=stack.efficiency())
    return dict(there=stack.propagate(state["field"], 0), back=stack.propagate(state["field"], 1, adjoint=True))


# ------------------------------------------------------------------ work
def work(case):
    """The method's own work: FFT operation counts (5 M log2 M per line; the N rows and the M columns
    of each padded transform), 6 per spectral product, ~30 per modulated pixel; bytes of the inputs,
    the outputs, and one read of the transfer table's quadrant per channel and distinct gap."""
    n, m, k, w, f = case["n"], case["m"], case["layers"], case["channels"], case["fov"]
    prop = (2 * n + 2 * m) * 5.0 * m * math.log2(m) + 6.0 * m * m
    quadrant = 8.0 * (m // 2 + 1) ** 2
    if case["kind"] == "propagate":
        return dict(bytes=w * (4 * 8.0 * n * n + quadrant), flops=2.0 * w * prop)
    tables = quadrant * ((k + 1) if case["unequal"] else 1)
    out = w * (4.0 * f * f * 2 + tables)
    if case["kind"] == "evaluate":
        return dict(bytes=out + 4.0 * k * n * n, flops=w * (k * prop + 30.0 * k * n * n))
    return dict(bytes=out + 8.0 * k * n * n, flops=w * (2.0 * k * prop + 60.0 * k * n * n))


# ------------------------------------------------------------------ the method in 64 bits
def _transfer(c, d, lam, g, shift, dev):
    """[channels][M][M] transfer function of gap g, with displaced layers' phase ramps."""
    m = c["m"]
    fr = torch.fft.fftfreq(m, d=float(d["pitch"]), dtype=torch.float64, device=dev)
    fy, fx = fr[:, None], fr[None, :]
    z = float(d["gaps"][g])
    ramp = None
    if shift is not None:
        at = lambda l: shift[l - 1] if 1 <= l <= c["layers"] else np.zeros(3)  # noqa: E731
        a = at(g) - at(g + 1)
        z += float(at(g + 1)[2] - at(g)[2])
        ramp = -2.0 * math.pi * (fx * float(a[0]) + fy * float(a[1]))
    q = (c["medium"] / lam[:, None, None]) ** 2 - fx * fx - fy * fy
    root = q.abs().sqrt()
    H = torch.polar(torch.ones_like(q), 2.0 * math.pi * z * root)
    gone = torch.exp(-2.0 * math.pi * z * root) if c["evanescent"] == "decay" else torch.zeros_like(q)
    H = torch.where(q >= 0, H, gone.to(H.dtype))
    return H if ramp is None else H * torch.polar(torch.ones_like(ramp), ramp)


def _gap(u, H, n, m, adjoint=False):
    o = (m - n) // 2
    p = torch.nn.functional.pad(torch.view_as_real(u), (0, 0, o, m - n - o, o, m - n - o))
    s = torch.fft.fft2(torch.view_as_complex(p.contiguous())) * (H.conj() if adjoint else H)
    return torch.fft.ifft2(s)[:, o:o + n, o:o + n]


def exact(case, seed):
    c, d, s = case, _design(case), _inputs(case, seed)
    n, m, k, f = c["n"], c["m"], c["layers"], c["fov"]
    if (1 if c["kind"] == "evaluate" else 3) * c["channels"] * (k + 1) * m * m > 2.0e10:
        return None
    some = max(1, int(2.0e7 / (m * m * (1 if c["kind"] in ("propagate", "evaluate") else k + 1))))
    parts = [slice(i, min(i + some, c["channels"])) for i in range(0, c["channels"], some)]
    dev = (s["field"] if "field" in s else s["h"]).device
    lams = torch.tensor(d["lam"], dtype=torch.float64, device=dev)
    if c["kind"] == "propagate":
        there = torch.empty((c["channels"], n, n), dtype=torch.complex128, device=dev)
        back = torch.empty_like(there)
        for p in parts:
            u = s["field"][p].to(torch.complex128)
            there[p] = _gap(u, _transfer(c, d, lams[p], 0, None, dev), n, m)
            back[p] = _gap(u, _transfer(c, d, lams[p], 1, None, dev), n, m, adjoint=True)
        return dict(there=there, back=back)
    h32 = s["h"]
    if c["kind"] == "evaluate":  # the levels as they are documented: the index decided in 32 bits
        levels, h_max = float(2 ** c["bits"] - 1), float(d["lam_m"])
        scale, step = np.float32(levels / h_max), np.float32(h_max / levels)
        h32 = torch.round(h32.clamp(0.0, float(np.float32(h_max))) * float(scale)) * float(step)
    h = h32.detach().to(torch.float64)
    learn = c["kind"] != "evaluate"
    T = s["T"].to(torch.float64)
    n_index = torch.tensor(d["n_index"], dtype=torch.float64, device=dev)
    fd, of, norm = f // c["bin"], (n - f) // 2, float(c["channels"]) * (f // c["bin"]) ** 2
    I_all = torch.empty((c["channels"], f, f), dtype=torch.float64, device=dev)
    psnr = torch.empty(c["channels"], dtype=torch.float64, device=dev)
    grad = torch.zeros_like(h)
    loss = torch.zeros((), dtype=torch.float64, device=dev)
    u0 = torch.zeros((n, n), dtype=torch.complex128, device=dev)
    u0[of:of + f, of:of + f] = 1.0
    for p in parts:
        lam, hp = lams[p], h.clone().requires_grad_(learn)
        with torch.set_grad_enabled(learn):
            v = _gap(u0.expand(lam.shape[0], n, n), _transfer(c, d, lam, 0, s.get("shift"), dev), n, m)
            for l in range(1, k + 1):
                x = (hp[l - 1] + c["base"] * NM)[None] / lam[:, None, None]
                t = torch.polar(torch.exp(-2.0 * math.pi * c["kappa"] * x),
                                -2.0 * math.pi * (n_index[p] - c["medium"])[:, None, None] * x)
                v = _gap(t * v, _transfer(c, d, lam, l, s.get("shift"), dev), n, m)
            o = v[:, of:of + f, of:of + f]
            I = o.real ** 2 + o.imag ** 2
            D = I.reshape(-1, fd, c["bin"], fd, c["bin"]).sum((2, 4))
            sigma = ((D * T[p]).sum((1, 2)) / (D * D).sum((1, 2))).detach()[:, None, None]
            scaled = (sigma * D - T[p]) ** 2
            part = (scaled if c["loss"] == "mse_scaled" else (D - T[p]) ** 2).sum() / norm
            if learn:
                grad += torch.autograd.grad(part, hp)[0]
        loss += part.detach()
        I_all[p] = I.detach()
        psnr[p] = -10.0 * torch.log10(scaled.detach().mean((1, 2)))
    if c["kind"] == "evaluate":
        return dict(I=I_all, psnr=psnr, efficiency=I_all.sum((1, 2)) / float(f * f))
    return dict(grad=grad, I=I_all, loss=loss) if c["kind"] == "autograd" else dict(grad=grad, I=I_all, psnr=psnr)
