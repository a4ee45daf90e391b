"""The register sweeps of 64 x 64 and 128 x 128 windows, which FP16 amplitudes
take from 180 and 72 windows on (agent_impl), each call checked to run them: the
forward transform alone, absent probe values, the residual sums with the
pattern scale, readout and state between calls, graph replay, a caller's
capture, several jobs in one launch, the bounds-checking build, and runs of 100
iterations against the same iterations in 64 bits."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2111_14240_gb300 import datagen
from tests.gpu_helpers import TOL_ITER, TOL_NRMSE_REL, random_start, rel_l2, rounded_inputs, run_gpu, run_oracle
from tests.test_gpu_register_sweep import _workload

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SIZES = [(64, 180), (64, 609), (128, 72), (128, 153)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2111_14240_gb300 import build
    build.build()


def _is_register_sweep(plan, np_):
    return plan["cluster"] == 1 and plan["threads"] == np_ * np_ // 32


def _job(w, init=None, graphs=True):
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    _, _, probe32, y32 = rounded_inputs(w)
    codes, scales = datagen.quantize_amplitudes_f16(y32.astype(np.float64))
    old = os.environ.get("PMACE_GRAPHS")
    os.environ["PMACE_GRAPHS"] = "1" if graphs else "0"
    try:
        rec = pm.Reconstruction(probe32, w.offsets, torch.from_numpy(codes).cuda(), w.x.shape,
                                amp_format=pm.PMACE_AMP_F16_SCALED, scales=torch.from_numpy(scales).cuda(), init=init)
    finally:
        if old is None:
            os.environ.pop("PMACE_GRAPHS", None)
        else:
            os.environ["PMACE_GRAPHS"] = old
    assert _is_register_sweep(rec.plan(), w.np_)
    return rec


@pytest.mark.parametrize("np_,J,f16,taken", [(64, 179, True, False), (64, 180, True, True), (64, 400, False, False),
                                             (128, 71, True, False), (128, 72, True, True), (128, 200, False, False),
                                             (32, 1, False, True), (32, 1, True, True), (256, 80, True, False)])
def test_which_jobs_take_the_register_sweep(np_, J, f16, taken):
    plan = run_gpu(_workload(np_, J), 0, 0.5, f16=f16, want_patches=False)["plan"]
    if np_ == 32:
        assert taken == (plan["cluster"] == 1 and plan["threads"] == 128)
    else:
        assert taken == _is_register_sweep(plan, np_) and (taken or plan["cluster"] == np_ // 16)


@pytest.mark.parametrize("np_,J", SIZES)
def test_forward_transform(np_, J):
    """As test_forward_transform_stage_matches_fft, with its bar."""
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    w = _workload(np_, J, absent=True)
    x0 = random_start(w)
    rec = _job(w, x0)
    out = torch.empty((J, np_, np_, 2), dtype=torch.float32, device="cuda")
    pm.pmace_debug_spectra(rec.h, 0.5, 0.5, out)
    got = torch.view_as_complex(out).cpu().numpy().astype(np.complex128) / np_
    rec.close()
    v = np.stack([x0[r:r + np_, c:c + np_] for r, c in w.offsets]).astype(np.complex128)
    ref = np.fft.fft2(w.probe.astype(np.complex64).astype(np.complex128)[None] * v, norm="ortho")
    assert rel_l2(got, ref) < 2e-6


@pytest.mark.parametrize("np_,J", SIZES)
@pytest.mark.parametrize("rho", [0.4, 0.5])
def test_absent_probe_values_and_residuals(np_, J, rho):
    """Pixels whose probe value is 0 return the agent's input; r_fp and r_data
    of the first and of the second iteration."""
    w = _workload(np_, J, absent=True)
    x0 = random_start(w)
    for n in (1, 2):
        g, o = run_gpu(w, n, 0.5, rho, f16=True, init=x0), run_oracle(w, n, 0.5, rho, f16=True, x0=x0)
        assert _is_register_sweep(g["plan"], np_)
        assert rel_l2(g["x_hat"], o["x_hat"]) < n * TOL_ITER
        assert rel_l2(g["v"], o["v"]) < n * TOL_ITER
        assert abs(g["r_data"] / o["r_data"] - 1) < 1e-4
        assert abs(g["r_fp"] / o["r_fp"] - 1) < 1e-4


@pytest.mark.parametrize("np_,J", [(64, 190), (128, 90)])
def test_rho_switches_state_graphs_and_capture(np_, J):
    """rho on both sides of 1/2 in one run, the image read between the calls;
    a state saved and resumed; replayed graphs against direct launches; a
    call captured by the caller: all bit for bit."""
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    w = _workload(np_, J)
    x0 = random_start(w)
    steps = [(1, 0.5, 0.5), (2, 0.5, 0.3), (1, 0.7, 0.8), (13, 0.4, 0.4), (12, 0.4, 0.6)]
    rec, direct, resumed = _job(w, x0), _job(w, x0, graphs=False), _job(w)
    q = torch.empty((J, np_, np_, 2), device="cuda")
    xb = torch.empty((*w.x.shape, 2), device="cuda")
    for k, (n, alpha, rho) in enumerate(steps):
        for r in (rec, direct) + ((resumed,) if k > 1 else ()):
            r.iterate(n, alpha, rho)
        want = rec.image().cpu().numpy()
        assert np.array_equal(direct.image().cpu().numpy(), want) and direct.residual() == rec.residual()
        if k == 1:
            info = pm.pmace_get_state(rec.h, q, xb)
            pm.pmace_set_state(resumed.h, q, xb, info)
        if k >= 1:
            assert np.array_equal(resumed.image().cpu().numpy(), want)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rec.iterate(1, 0.4, 0.6)
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        direct.iterate(1, 0.4, 0.6)
        assert np.array_equal(rec.image().cpu().numpy(), direct.image().cpu().numpy())
    for r in (rec, direct, resumed):
        r.close()


def test_several_jobs_in_one_launch():
    """Served together, jobs of both sizes equal the plain call bit for bit."""
    from paper_2111_14240_gb300 import pmace as pm
    srv, jobs = pm.Server(), []
    for k, (np_, J) in enumerate([(64, 180), (128, 72), (64, 301), (128, 160), (128, 75)]):
        w = _workload(np_, J, seed=k)
        _, _, probe32, y32 = rounded_inputs(w)
        codes, scales = datagen.quantize_amplitudes_f16(y32.astype(np.float64))
        rho = (0.5, 0.4, 0.6)[k % 3]
        jobs.append((w, rho, srv.submit(probe32, w.offsets, codes, w.x.shape, 3 + k, 0.5, rho,
                                        amp_format=pm.PMACE_AMP_F16_SCALED, scales=scales)))
    for k, (w, rho, jid) in enumerate(jobs):
        res, img = srv.wait(jid)
        assert res["status"] == 0, res
        rec = _job(w)
        rec.iterate(3 + k, 0.5, rho)
        assert np.array_equal(img, rec.image().cpu().numpy()), k
        rec.close()
    srv.close()


SCRIPT = r"""
import json, sys
import numpy as np
from paper_2111_14240_gb300 import pmace as pm
from tests.test_gpu_register_sweep import _workload
from tests.test_gpu_register_sweep_f16 import _job
status, imgs = [], []
for np_, J in ((64, 190), (128, 75)):
    rec = _job(_workload(np_, J))
    rec.iterate(3, 0.5, 0.5)
    st = 0
    try:
        rec.residual()
        img = np.empty((rec.n1, rec.n2), np.complex64)
        pm.pmace_get_image(rec.h, img)
        imgs.append(img)
    except pm.PmaceError as e:
        st = e.status
    status.append(st)
    rec.close()
if imgs:
    np.save(sys.argv[1], np.concatenate([i.ravel() for i in imgs]))
print(json.dumps({"library": pm._LIB_PATH, "status": status}))
"""


def test_bounds_checking_build(tmp_path):
    """The same images from the bounds-checking build; a window corner
    overwritten with one past the image is clamped and reported."""
    from paper_2111_14240_gb300 import build
    from paper_2111_14240_gb300 import pmace as pm
    debug = build.build_debug()
    out = {}
    for name, env in (("release", {}), ("debug", {"PMACE_LIBRARY": debug}),
                      ("inject", {"PMACE_LIBRARY": debug, "PMACE_INJECT_BAD_OFFSET": "1"})):
        path = str(tmp_path / f"{name}.npy")
        base = {k: v for k, v in os.environ.items() if k not in ("PMACE_LIBRARY", "PMACE_INJECT_BAD_OFFSET")}
        r = subprocess.run([sys.executable, "-c", SCRIPT, path], cwd=ROOT, env={**base, **env}, capture_output=True,
                           text=True, timeout=600)
        assert r.returncode == 0, r.stderr[-3000:]
        res = json.loads([ln for ln in r.stdout.splitlines() if ln.startswith("{")][-1])
        assert ("debug" in os.path.basename(res["library"])) == bool(env)
        out[name] = res["status"], np.load(path) if os.path.exists(path) else None
    assert out["release"][0] == out["debug"][0] == [0, 0]
    assert np.array_equal(out["release"][1], out["debug"][1])
    assert out["inject"][0] == [pm.PMACE_ERR_STATE] * 2


def _run64(y, probe, offsets, shape, alpha, rho, kappa, counts):
    """Algorithm 1 in complex128 with torch: the readout at each count, and Lambda."""
    import torch
    n, (n1, n2), J = probe.shape[0], shape, offsets.shape[0]
    o, i = torch.from_numpy(offsets.astype(np.int64)).cuda(), torch.arange(n, device="cuda")
    idx = (o[:, 0, None, None] + i[None, :, None]) * n2 + o[:, 1, None, None] + i[None, None, :]
    d, y = torch.from_numpy(probe).cuda(), torch.from_numpy(y).cuda()
    wk = d.abs() ** kappa

    def add(stack, k):
        out = torch.zeros((n1 * n2, k), dtype=torch.float64, device="cuda")
        return out.index_add_(0, idx.reshape(-1), stack.reshape(-1, k))

    lam = add(wk.expand(J, n, n), 1)[:, 0]
    inv = torch.where(lam > 0, 1.0 / lam, torch.zeros_like(lam))

    def average(stack):
        return torch.view_as_complex(add(torch.view_as_real(stack * wk), 2)) * inv

    c = torch.sqrt((y * y).sum() / (J * (d.abs() ** 2).sum()))
    v = torch.zeros((J, n, n), dtype=torch.complex128, device="cuda") + c
    images = []
    for it in range(1, counts[-1] + 1):
        f = torch.fft.fft2(d * v, norm="ortho")
        m = f.abs()
        g = torch.fft.ifft2(torch.where(m > 0, y / m, torch.zeros_like(m)) * f, norm="ortho")
        w = (alpha * v + g / d) / (1 + alpha)
        z = average(2 * w - v)
        v = v + 2 * rho * (z[idx] - w)
        if it in counts:
            images.append(average(v).reshape(n1, n2).cpu().numpy())
    return images, lam.reshape(n1, n2).cpu().numpy()


GEO = {128: dict(n_obj=600, n_p=128, probe_sigma=32.0, n_scan=30, step=16, jitter=2, name="c30"),
       64: dict(n_obj=560, n_p=64, probe_sigma=16.0, n_scan=30, step=16, jitter=2, name="c30_64")}


@pytest.mark.parametrize("np_,peak,alpha", [(128, 1e4, 0.5), (128, 1e6, 0.5), (128, 1e4, 2.0), (128, 1e6, 2.0),
                                            (64, 1e4, 0.5), (64, 1e6, 2.0)])
def test_hundred_iterations_track_64_bits_on_the_decoded_codes(np_, peak, alpha):
    """The reconstruction error of a converging geometry (900 windows) from the
    constant start, every ten iterations, within 1 % of that of the 64-bit run
    on the amplitudes the codes stand for (so without their 2^-11 steps):
    128 x 128 windows on the covered and on the well-illuminated pixels
    (Lambda at least a tenth of its peak), 64 x 64 windows, whose larger share
    of edge pixels the data do not determine, on the latter."""
    from oracle import pmace_oracle as orc
    w = datagen.make_workload(GEO[np_], seed=1, peak=peak)
    counts = list(range(10, 101, 10))
    _, _, probe32, y32 = rounded_inputs(w)
    codes, scales = datagen.quantize_amplitudes_f16(y32.astype(np.float64))
    images, lam = _run64(datagen.dequantize_f16(codes, scales), probe32.astype(np.complex128), w.offsets, w.x.shape,
                         alpha, 0.5, 1.25, counts)
    masks = [lam >= 0.1 * lam.max()] + ([lam > 0] if np_ == 128 else [])
    rec, done = _job(w), 0
    for k, ref in zip(counts, images):
        rec.iterate(k - done, alpha, 0.5)
        done = k
        got = rec.image().cpu().numpy().astype(np.complex128)
        for m in masks:
            e, e64 = orc.nrmse(got, w.x, m), orc.nrmse(ref, w.x, m)
            assert abs(e - e64) <= TOL_NRMSE_REL * e64, (k, e, e64)
    rec.close()
