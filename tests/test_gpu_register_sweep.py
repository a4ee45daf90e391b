"""The register sweeps (agent_reg.cuh: a window a warp for 32 x 32 probes, a
CTA for 64 x 64 and 128 x 128), the consensus taken from the pending stack, and
the readout image kept with the state, against the FP64 oracle: window counts
at the edges of the dispatch rules, remainders of the windows a CTA takes, both
amplitude formats, and step parameters on both sides of rho = 1/2."""
import numpy as np
import pytest

from tests.gpu_helpers import TOL_ITER, random_start, rel_l2, run_gpu, run_oracle

pytestmark = pytest.mark.gpu


def _workload(np_, J, seed=1, absent=False):
    """J windows at random corners of a non-square image, amplitudes of a
    random object (no noise: only the arithmetic is compared)."""
    from paper_2111_14240_gb300 import datagen

    rng = np.random.Generator(np.random.PCG64(seed))
    n1, n2 = np_ + 37, np_ + 61 + J // 8
    x = datagen.make_object(rng, n1, n2)
    probe = datagen.make_probe(rng, np_, np_ / 4.0)
    if absent:
        probe[: np_ // 8, np_ // 2:] = 0.0
    offs = np.stack([rng.integers(0, n1 - np_ + 1, J), rng.integers(0, n2 - np_ + 1, J)], axis=1).astype(np.int32)
    y = datagen.simulate(None, x, probe, offs, None)
    return datagen.Workload(f"reg{np_}", x, probe, offs, y, None, seed)


# (probe, windows): one window, fewer than a CTA's four warps, one more than
# them, one round of the device and one more; the windows from which the
# register sweep takes over, one below and one above
CASES = [(32, 1), (32, 3), (32, 5), (32, 2433), (64, 179), (64, 180), (64, 609), (128, 71), (128, 72), (128, 153)]


@pytest.mark.parametrize("np_,J", CASES)
@pytest.mark.parametrize("f16,alpha,rho", [(False, 0.5, 0.5), (True, 2.0, 0.4), (True, 0.3, 0.7)])
def test_matches_oracle(np_, J, f16, alpha, rho):
    w = _workload(np_, J)
    x0 = random_start(w)
    g = run_gpu(w, 2, alpha, rho, f16=f16, init=x0)
    o = run_oracle(w, 2, alpha, rho, f16=f16, x0=x0)
    d = np.abs(w.probe)
    assert rel_l2(g["x_hat"], o["x_hat"]) < 2 * TOL_ITER
    assert rel_l2(g["v"] * d, o["v"] * d) < 2 * TOL_ITER
    assert rel_l2(g["v"], o["v"]) < 2 * TOL_ITER


@pytest.mark.parametrize("np_,J", [(32, 9), (64, 200), (128, 80)])
def test_absent_probe_values(np_, J):
    """Pixels whose probe value is 0 return the agent's input."""
    w = _workload(np_, J, absent=True)
    x0 = random_start(w)
    g, o = run_gpu(w, 1, 0.5, 0.5, init=x0), run_oracle(w, 1, 0.5, 0.5, x0=x0)
    assert rel_l2(g["x_hat"], o["x_hat"]) < TOL_ITER
    assert rel_l2(g["v"], o["v"]) < TOL_ITER


@pytest.mark.parametrize("np_,J", [(32, 40), (64, 190), (128, 75)])
def test_residuals_match_oracle_quantities(np_, J):
    """r_fp and r_data of the second iteration."""
    w = _workload(np_, J)
    x0 = random_start(w)
    alpha, rho = 0.5, 0.5
    g = run_gpu(w, 2, alpha, rho, init=x0)
    o = run_oracle(w, 2, alpha, rho, x0=x0)
    assert abs(g["r_data"] / o["r_data"] - 1) < 1e-4
    assert abs(g["r_fp"] / o["r_fp"] - 1) < 1e-4


@pytest.mark.parametrize("np_,J", [(32, 169), (64, 81), (128, 90), (256, 4)])
def test_rho_switches_state_and_readout(np_, J):
    """Calls with rho on both sides of 1/2 in one run (the consensus comes from
    u and from q in turn), the image read between them, and a state saved,
    replaced and resumed, bit for bit."""
    import torch

    from paper_2111_14240_gb300 import pmace as pm

    w = _workload(np_, J)
    x0 = random_start(w)
    steps = [(1, 0.5, 0.5), (2, 0.5, 0.3), (1, 0.7, 0.8), (1, 0.7, 0.4), (2, 0.4, 0.6)]
    rec = pm.Reconstruction(w.probe.astype(np.complex64), w.offsets, w.y.astype(np.float32), w.x.shape, init=x0)
    q = torch.empty((w.J, np_, np_, 2), device="cuda")
    xb = torch.empty((*w.x.shape, 2), device="cuda")
    images, info = [], None
    for k, (n, alpha, rho) in enumerate(steps):
        rec.iterate(n, alpha, rho)
        images.append(rec.image().cpu().numpy())
        if k == 1:
            info = pm.pmace_get_state(rec.h, q, xb)
    # the readout without the kept image: the same state in a new job
    again = pm.Reconstruction(w.probe.astype(np.complex64), w.offsets, w.y.astype(np.float32), w.x.shape)
    pm.pmace_set_state(again.h, q, xb, info)
    assert np.array_equal(again.image().cpu().numpy(), images[1])
    for (n, alpha, rho), want in zip(steps[2:], images[2:]):
        again.iterate(n, alpha, rho)
        assert np.array_equal(again.image().cpu().numpy(), want)
    # a state put back into a job that has moved on
    pm.pmace_set_state(rec.h, q, xb, info)
    rec.iterate(*steps[2])
    assert np.array_equal(rec.image().cpu().numpy(), images[2])
    rec.close()
    again.close()
    state = None
    for n, alpha, rho in steps[:2]:
        o = run_oracle(w, n, alpha, rho, x0=x0) if state is None else run_oracle(w, n, alpha, rho, v0=state["v"],
                                                                                z_prev=state["z"])
        state = o
    assert rel_l2(images[1].astype(np.complex128), state["x_hat"]) < 3 * TOL_ITER


@pytest.mark.parametrize("np_,J", [(32, 40), (128, 80)])
def test_iteration_captured_by_the_caller(np_, J):
    """An iterate call captured in the caller's graph and replayed after the
    state was replaced gives what the call gives."""
    import torch

    from paper_2111_14240_gb300 import pmace as pm

    w = _workload(np_, J)
    rec = pm.Reconstruction(w.probe.astype(np.complex64), w.offsets, w.y.astype(np.float32), w.x.shape,
                            init=random_start(w))
    rec.iterate(2, 0.5, 0.5)
    q = torch.empty((w.J, np_, np_, 2), device="cuda")
    xb = torch.empty((*w.x.shape, 2), device="cuda")
    info = pm.pmace_get_state(rec.h, q, xb)
    rec.iterate(1, 0.5, 0.5)
    want = rec.image().cpu().numpy()
    rec.iterate(3, 0.5, 0.5)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rec.iterate(1, 0.5, 0.5)
    pm.pmace_set_state(rec.h, q, xb, info)
    graph.replay()
    torch.cuda.synchronize()
    got = rec.image().cpu().numpy()
    rec.close()
    assert np.array_equal(got, want)
