"""What a user of the framework has it do, as cases that can be timed.

Four uses, each through the public binding (paper_2111_14240_gb300.pmace):

* iterate:  a reconstruction resident on the GPU is advanced by some
            iterations and its image read back on the device, optionally with
            the patch stack or the residuals: the steady work of every job;
* job:      a whole job from host arrays: create, iterate, image to the host;
* serve:    a batch of jobs of mixed sizes submitted to a running server;
* simulate: measured amplitudes of a known object (forward model and Poisson
            noise), host arrays in and out.

Problems are drawn as the repository's workloads are: a random object
(amplitude U[0.6, 1], phase U[0, pi/2], here without the smoothing), a
Gaussian probe of sigma Np / 4 with a random quadratic phase, a jittered
raster scan, Poisson noise at a peak count.  Reconstructions start from a
rough earlier result (the object with 2 % noise), from which every spectral
coefficient is resolved in single precision; a pass runs a few iterations,
over which single-precision runs stay comparable.
"""
import math

import numpy as np
import torch

from paper_2111_14240_gb300 import pmace as pm

# case fields: use, image n1 x n2, probe side np, raster s1 x s2 with step and
# jitter, f16 (amplitude codes with per-pattern scales), photon peak, iters
# (iterations of one pass), alpha, rho, kappa, outputs beside the image
_ITER = dict(use="iterate", jitter=2, f16=False, peak=1e5, alpha=0.5, rho=0.5, kappa=1.25, outputs="image")


def listed():
    c = []

    def add(name, **k):
        c.append(dict(_ITER, **k, name=name))

    # the smallest configuration (128^2 object, 32 px probe, 169 windows), with the
    # residuals of a user's progress loop: launches and latency
    add("p32_small", n1=128, n2=128, np=32, s1=13, s2=13, step=8, jitter=1, iters=2, outputs="residual")
    # the same probe on a scan that fills the GPU, FP16 amplitudes
    add("p32_wide", n1=512, n2=512, np=32, s1=60, s2=60, step=8, jitter=1, f16=True, iters=2)
    # a small 64 px scan, patch stack read back too
    add("p64_small", n1=200, n2=200, np=64, s1=9, s2=9, step=16, iters=2, outputs="patches")
    # a 64 px scan of the serving distribution's largest object
    add("p64_wide", n1=1024, n2=1024, np=64, s1=60, s2=60, step=16, f16=True, iters=2)
    # the converging 128 px raster (900 windows), FP32 amplitudes
    add("p128_900", n1=600, n2=600, np=128, s1=30, s2=30, step=16, peak=1e6, iters=2, outputs="residual")
    # odd sizes: a non-square image, a window count that divides by nothing, other step parameters
    add("p128_ragged", n1=517, n2=771, np=128, s1=19, s2=31, step=19, iters=2, alpha=2.0, rho=0.4, kappa=2.0)
    # the 2048^2 precision workload: 14641 windows, FP16 amplitudes
    add("p128_wide", n1=2048, n2=2048, np=128, s1=121, s2=121, step=16, peak=1e6, f16=True, iters=2)
    # the largest single scan: 8192^2, 64009 windows, FP16 amplitudes
    add("p128_large", n1=8192, n2=8192, np=128, s1=253, s2=253, step=32, jitter=3, f16=True, iters=2)
    # the 256 px probe workload, 324 windows
    add("p256", n1=600, n2=600, np=256, s1=18, s2=18, step=20, iters=2)
    # a whole job from host arrays to a host image
    add("job_p128", use="job", n1=512, n2=512, np=128, s1=24, s2=24, step=16, peak=1e6, f16=True, iters=2)
    # a batch of mixed jobs on a running server
    add("serve", use="serve", n1=512, n2=512, np=128, s1=24, s2=24, step=16, f16=True, iters=2, jobs=12)
    # the data simulator, 64 px
    add("simulate", use="simulate", n1=512, n2=512, np=64, s1=28, s2=28, step=16)
    return c


def _fits(c, most=64009 * 128 * 128 * 2):
    return c["s1"] * c["s2"] * c["np"] ** 2 * c["iters"] <= most


def draw(rng):
    while True:
        c = dict(_ITER)
        c["use"] = rng.choice(["iterate"] * 7 + ["job", "serve", "simulate"])
        c["np"] = rng.choice([32, 64, 128, 128, 256])
        c["step"] = rng.randint(8, 32) if c["np"] >= 64 else rng.randint(4, 12)
        c["jitter"] = rng.randint(0, 3)
        most = {32: 160, 64: 160, 128: 200, 256: 24}[c["np"]] if c["use"] == "iterate" else 24
        c["s1"] = int(round(math.exp(rng.uniform(math.log(3), math.log(most)))))
        c["s2"] = max(2, int(round(c["s1"] * rng.uniform(0.6, 1.4))))
        c["n1"] = c["np"] + (c["s1"] - 1) * c["step"] + rng.randint(2, 40)
        c["n2"] = c["np"] + (c["s2"] - 1) * c["step"] + rng.randint(2, 40)
        c["f16"] = rng.random() < 0.5
        c["peak"] = 10.0 ** rng.randint(5, 6)
        c["alpha"] = rng.choice([0.3, 0.5, 0.7, 1.0, 2.0])
        c["rho"] = rng.choice([0.5, 0.5, 0.5, 0.3, 0.6])
        c["kappa"] = rng.choice([1.25, 1.25, 2.0])
        c["iters"] = rng.randint(1, 2)
        if c["use"] == "iterate":
            c["outputs"] = rng.choice(["image", "image", "residual", "patches"])
        if c["use"] == "serve":
            c["np"], c["jobs"] = rng.choice([64, 128]), rng.randint(3, 12)
            c["n1"], c["n2"] = max(c["n1"], 160), max(c["n2"], 160)
            c["iters"] = rng.randint(1, 2)
        if c["n1"] <= 8192 and c["n2"] <= 8192 and _fits(c):
            return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _image(g, n1, n2):
    a = 0.6 + 0.4 * torch.rand((n1, n2), generator=g, device="cuda")
    p = 0.5 * math.pi * torch.rand((n1, n2), generator=g, device="cuda")
    return torch.polar(a, p)


def _problem(c, seed):
    """Object, start image, probe (complex64, GPU), offsets (int32, host)."""
    g = _gen(seed)
    n, rng = c["np"], np.random.Generator(np.random.PCG64(int(seed)))
    obj = _image(g, c["n1"], c["n2"])
    noise = torch.randn((2, c["n1"], c["n2"]), generator=g, device="cuda")
    init = obj + 0.02 * torch.complex(noise[0], noise[1])
    r = torch.arange(n, device="cuda", dtype=torch.float64) - (n - 1) / 2
    r2 = r[:, None] ** 2 + r[None, :] ** 2
    sigma = n / 4
    probe = torch.polar(torch.exp(-r2 / (2 * sigma * sigma)), rng.uniform(0, 2 * math.pi) * r2 / (n / 2) ** 2)
    offs = np.empty((c["s1"] * c["s2"], 2), np.int32)
    for ax, (side, count) in enumerate(((c["n1"], c["s1"]), (c["n2"], c["s2"]))):
        k = np.arange(c["s1"] * c["s2"])
        k = k // c["s2"] if ax == 0 else k % c["s2"]
        base = (side - (count - 1) * c["step"] - n) // 2 + k * c["step"]
        offs[:, ax] = np.clip(base + rng.integers(-c["jitter"], c["jitter"] + 1, k.size), 0, side - n)
    return obj, init, probe.to(torch.complex64), offs


def _chunks(J, n):
    step = max(1, (1 << 26) // (n * n))
    return [(a, min(J, a + step)) for a in range(0, J, step)]


def _index(offs, n, n2, a, b):
    """Flat image indices of the windows a .. b - 1, (b - a, n, n)."""
    o = torch.from_numpy(offs[a:b].astype(np.int64)).cuda()
    i = torch.arange(n, device="cuda")
    return (o[:, 0, None, None] + i[None, :, None]) * n2 + o[:, 1, None, None] + i[None, None, :]


def _measured(c, seed, obj, probe, offs):
    """Amplitudes with Poisson noise on the GPU: (float32, None) or (FP16 codes, scales)."""
    g, n, J = _gen(seed + 1), c["np"], offs.shape[0]
    out = torch.empty((J, n, n), dtype=torch.float16 if c["f16"] else torch.float32, device="cuda")
    scales = torch.empty(J, dtype=torch.float32, device="cuda") if c["f16"] else None
    for a, b in _chunks(J, n):
        w = torch.fft.fft2(obj.reshape(-1)[_index(offs, n, c["n2"], a, b)] * probe, norm="ortho")
        inten = w.real.square() + w.imag.square()
        r = c["peak"] / inten.amax(dim=(1, 2), keepdim=True)
        y = torch.sqrt(torch.poisson(inten * r, generator=g) / r)
        if c["f16"]:
            scales[a:b] = y.amax(dim=(1, 2))
            y = y / scales[a:b, None, None]
        out[a:b] = y
    return out, scales


def _fmt(c):
    return pm.PMACE_AMP_F16_SCALED if c["f16"] else pm.PMACE_AMP_F32


def _jobs(c, seed):
    """The mixed jobs of a served batch: smaller and larger scans of both probe sizes."""
    out = []
    for k in range(c["jobs"]):
        j = dict(c, use="iterate", np=(64, c["np"])[k % 2], alpha=(0.3, 0.5, 1.0)[k % 3], peak=10.0 ** (5 + k % 2))
        j["s1"], j["s2"] = max(3, c["s1"] - 2 * (k % 5)), max(3, c["s2"] - 3 * (k % 4))
        j["step"] = max(4, (min(j["n1"], j["n2"]) - j["np"]) // max(j["s1"], j["s2"], c["s1"]))
        out.append((j, seed * 100 + k))
    return out


def _host_job(c, seed):
    obj, init, probe, offs = _problem(c, seed)
    y, scales = _measured(c, seed, obj, probe, offs)
    return dict(case=c, probe=probe.cpu().numpy(), offs=offs, y=y.cpu().numpy(),
                scales=None if scales is None else scales.cpu().numpy(), init=init.cpu().numpy())


# ------------------------------------------------------------------- passes
def prepare(case, seed):
    c = case
    if c["use"] == "serve":
        return dict(case=c, server=pm.Server(), jobs=[_host_job(j, s) for j, s in _jobs(c, seed)])
    if c["use"] == "simulate":
        obj, _, probe, offs = _problem(c, seed)
        return dict(case=c, obj=obj.cpu().numpy(), probe=probe.cpu().numpy(), offs=offs, seed=int(seed))
    if c["use"] == "job":
        return _host_job(c, seed)
    obj, init, probe, offs = _problem(c, seed)
    y, scales = _measured(c, seed, obj, probe, offs)
    rec = pm.Reconstruction(probe, offs, y, (c["n1"], c["n2"]), kappa=c["kappa"], amp_format=_fmt(c),
                            scales=scales, init=init)
    return dict(case=c, rec=rec)


def run(state):
    c = state["case"]
    if c["use"] == "serve":
        s, ids = state["server"], []
        for j in state["jobs"]:
            k = j["case"]
            ids.append(s.submit(j["probe"], j["offs"], j["y"], (k["n1"], k["n2"]), k["iters"], k["alpha"], k["rho"],
                                k["kappa"], _fmt(k), j["scales"], j["init"]))
        out = [s.wait(i)[1] for i in ids]
        for i in ids:
            s.release(i)
        return out
    if c["use"] == "simulate":
        return pm.simulate(state["obj"], state["probe"], state["offs"], peak=c["peak"], seed=state["seed"])
    if c["use"] == "job":
        rec = pm.Reconstruction(state["probe"], state["offs"], state["y"], (c["n1"], c["n2"]), kappa=c["kappa"],
                                amp_format=_fmt(c), scales=state["scales"], init=state["init"])
        rec.iterate(c["iters"], c["alpha"], c["rho"])
        out = rec.image().cpu()
        rec.close()
        return out
    rec = state["rec"]
    rec.iterate(c["iters"], c["alpha"], c["rho"])
    out = {"image": rec.image()}
    if c["outputs"] == "patches":
        out["patches"] = rec.patches()
    if c["outputs"] == "residual":
        out["residual"] = list(rec.residual())
    return out


def work(case):
    """One pass: per iteration every stack value read and written once, every
    amplitude read once, the consensus image read and written once, and two
    2-D transforms a window (5 P log2 P operations each, P = Np^2) with about
    45 operations a pixel beside them."""
    c = case
    jobs = [j for j, _ in _jobs(c, 0)] if c["use"] == "serve" else [c]
    total, flops = 0.0, 0.0
    for j in jobs:
        P, J, NI = j["np"] ** 2, j["s1"] * j["s2"], j["n1"] * j["n2"]
        fft = 5.0 * P * math.log2(P)
        y = J * P * (2 if j["f16"] else 4)
        if c["use"] == "simulate":
            total += NI * 8 + J * P * 4
            flops += J * (fft + 20.0 * P)
            continue
        total += j["iters"] * (J * P * 16 + y + NI * 16) + NI * 8
        flops += j["iters"] * J * (2 * fft + 45.0 * P)
        if j["outputs"] == "patches":
            total += J * P * 8
        if c["use"] != "iterate":   # the inputs go to the device
            total += y + NI * 8
    return {"bytes": total, "flops": flops}


# -------------------------------------------------------------------- exact
def _reconstruct64(c, seed):
    """Algorithm 1 in complex128 on the inputs as the library gets them."""
    obj, init, probe, offs = _problem(c, seed)
    y16, scales = _measured(c, seed, obj, probe, offs)
    del obj
    n, n1, n2, J = c["np"], c["n1"], c["n2"], offs.shape[0]
    alpha, rho, kappa = (float(np.float32(c[k])) for k in ("alpha", "rho", "kappa"))
    d = probe.to(torch.complex128)
    wk = d.abs() ** kappa
    parts = _chunks(J, n)
    lam = torch.zeros(n1 * n2, dtype=torch.float64, device="cuda")
    x0 = init.to(torch.complex128).reshape(-1)
    v = torch.empty((J, n, n), dtype=torch.complex128, device="cuda")
    for a, b in parts:
        i = _index(offs, n, n2, a, b)
        lam.index_add_(0, i.reshape(-1), wk.expand(b - a, n, n).reshape(-1))
        v[a:b] = x0[i]
    inv = torch.where(lam > 0, 1.0 / lam, torch.zeros_like(lam))

    def average(part):
        """Lambda^-1 sum_j P_j^t |D|^kappa part(a, b)."""
        s = torch.zeros((n1 * n2, 2), dtype=torch.float64, device="cuda")
        for a, b in parts:
            s.index_add_(0, _index(offs, n, n2, a, b).reshape(-1), torch.view_as_real(part(a, b) * wk).reshape(-1, 2))
        return torch.view_as_complex(s) * inv

    w = torch.empty_like(v)
    z = None
    for it in range(c["iters"]):
        sums = torch.zeros(4, dtype=torch.float64, device="cuda")
        for a, b in parts:
            f = torch.fft.fft2(d * v[a:b], norm="ortho")
            y = y16[a:b].double() * (scales[a:b, None, None].double() if scales is not None else 1.0)
            m = f.abs()
            g = torch.fft.ifft2(torch.where(m > 0, y / m, torch.zeros_like(m)) * f, norm="ortho")
            w[a:b] = (alpha * v[a:b] + g / d) / (1 + alpha)
            if c["outputs"] == "residual" and it + 1 == c["iters"]:
                zp = v[a:b] if z is None else z[_index(offs, n, n2, a, b)]
                for k, t in enumerate(((zp - w[a:b]).abs(), w[a:b].abs(), y - m, y)):
                    sums[k] += t.square().sum()
        z = average(lambda a, b: 2 * w[a:b] - v[a:b])
        for a, b in parts:
            v[a:b] += 2 * rho * (z[_index(offs, n, n2, a, b)] - w[a:b])
    out = {"image": average(lambda a, b: v[a:b]).reshape(n1, n2)}
    if c["outputs"] == "patches":
        out["patches"] = v
    if c["outputs"] == "residual":
        s = sums.tolist()
        out["residual"] = [math.sqrt(s[0] / s[1]), s[2] / s[3]]
    return out


def exact(case, seed):
    if case["use"] == "simulate":   # whole counts of a seeded generator: no value beside the library's own
        return None
    if case["use"] == "serve":
        return [_reconstruct64(j, s)["image"] for j, s in _jobs(case, seed)]
    out = _reconstruct64(case, seed)
    return out["image"] if case["use"] == "job" else out
