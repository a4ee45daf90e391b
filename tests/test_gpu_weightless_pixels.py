"""Pixels the probe does not weight: outside the scan the images read 0 whatever
a state that was set holds there."""
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
