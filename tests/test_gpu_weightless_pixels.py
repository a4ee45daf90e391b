"""Pixels the probe does not weight, or hardly: outside the scan the images read
0 whatever a state that was set holds there, and where Lambda is near the
smallest single-precision numbers an iteration stays finite."""
import numpy as np
import pytest

from tests.test_gpu_register_sweep import _workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("np_,J", [(32, 6), (64, 5)])
@pytest.mark.parametrize("rho", [0.3, 0.5, 0.7])
def test_uncovered_pixels_of_a_set_state_read_zero(np_, J, rho):
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    from tests.gpu_helpers import random_start
    w = _workload(np_, J)
    outside = np.ones(w.x.shape, bool)
    for r, c in w.offsets:
        outside[r:r + np_, c:c + np_] = False
    assert outside.any()
    out = []
    for fill in (0.0, 3.0, float("nan")):
        rec = pm.Reconstruction(w.probe.astype(np.complex64), w.offsets, w.y.astype(np.float32), w.x.shape,
                                init=random_start(w))
        rec.iterate(1, 0.5, rho)
        q = torch.empty((J, np_, np_, 2), device="cuda")
        xb = torch.empty((rec.n1, rec.n2, 2), device="cuda")
        info = pm.pmace_get_state(rec.h, q, xb)
        xb[torch.from_numpy(outside).cuda()] = fill
        pm.pmace_set_state(rec.h, q, xb, info)
        images = [rec.image().cpu().numpy()]
        for _ in range(2):
            rec.iterate(1, 0.5, rho)
            images.append(rec.image().cpu().numpy())
        pm.pmace_get_state(rec.h, q, xb)
        images.append(torch.view_as_complex(xb).cpu().numpy())
        rec.close()
        assert all((im[outside] == 0).all() for im in images), fill
        out.append(images)
    for images in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(images, out[0]))


@pytest.mark.parametrize("rho", [0.3, 0.5, 0.7])
def test_probe_tail_at_the_smallest_weights(rho):
    """|d|^2 = 4e-39 in two columns of the probe, alone there: Lambda^-1 is
    finite and (1/rho) Lambda^-1 is not.  The data say nothing about those
    pixels (1/d makes 1e11 of a rounding error), but they stay finite and the
    others are what the oracle gives."""
    from tests.gpu_helpers import TOL_ITER, random_start, rel_l2, run_gpu, run_oracle
    w = _workload(32, 1)
    w.probe[:, :2] = 6.3e-20
    x0 = random_start(w)
    g = run_gpu(w, 2, 0.5, rho, kappa=2.0, init=x0)
    o = run_oracle(w, 2, 0.5, rho, kappa=2.0, x0=x0)
    assert np.isfinite(g["x_hat"]).all() and np.isfinite(g["v"]).all()
    lit = np.abs(w.probe) > 0.1 * np.abs(w.probe).max()
    assert rel_l2(g["v"][:, lit], o["v"][:, lit]) < 2 * TOL_ITER
    (r, c), n = w.offsets[0], 32
    assert rel_l2(g["x_hat"][r:r + n, c:c + n][lit], o["x_hat"][r:r + n, c:c + n][lit]) < 2 * TOL_ITER
