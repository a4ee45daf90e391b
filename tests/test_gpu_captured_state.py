"""Calls that change a job's state, recorded in a caller's graph and replayed:
the image read after each replay, and an iteration launched after them, are
those of the same calls made directly, bit for bit."""
import numpy as np
import pytest

from tests.test_gpu_register_sweep import _workload

pytestmark = pytest.mark.gpu


def _job(np_, J):
    from paper_2111_14240_gb300 import pmace as pm
    from tests.gpu_helpers import random_start
    w = _workload(np_, J)
    return pm.Reconstruction(w.probe.astype(np.complex64), w.offsets, w.y.astype(np.float32), w.x.shape,
                             init=random_start(w))


def _host_image(rec):
    from paper_2111_14240_gb300 import pmace as pm
    img = np.empty((rec.n1, rec.n2), np.complex64)
    pm.pmace_get_image(rec.h, img)
    return img


def _captured(call):
    import torch
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call()

    def replay():
        graph.replay()
        torch.cuda.synchronize()
    return replay


@pytest.mark.parametrize("np_,J", [(32, 40), (128, 20)])
@pytest.mark.parametrize("rho", [0.3, 0.5, 0.7])
def test_image_after_every_replay_of_an_iteration(np_, J, rho):
    rec, ref = _job(np_, J), _job(np_, J)
    for r in (rec, ref):
        r.iterate(2, 0.5, rho)
    replay = _captured(lambda: rec.iterate(1, 0.5, rho))
    for _ in range(3):
        replay()
        ref.iterate(1, 0.5, rho)
        want = ref.image().cpu().numpy()
        assert np.array_equal(_host_image(rec), want)
        assert np.array_equal(rec.image().cpu().numpy(), want)
    replay()   # not read before the next iteration, whose consensus needs the readout image
    ref.iterate(1, 0.5, rho)
    for r in (rec, ref):
        r.iterate(1, 0.5, 0.5)
    assert np.array_equal(_host_image(rec), _host_image(ref))
    rec.close()
    ref.close()


@pytest.mark.parametrize("np_,J", [(32, 40), (128, 20)])
def test_image_after_every_replay_of_set_state(np_, J):
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    rec = _job(np_, J)
    rec.iterate(2, 0.5, 0.5)
    q = torch.empty((J, np_, np_, 2), device="cuda")
    xb = torch.empty((rec.n1, rec.n2, 2), device="cuda")
    info = pm.pmace_get_state(rec.h, q, xb)
    want = _host_image(rec)
    replay = _captured(lambda: pm.pmace_set_state(rec.h, q, xb, info))
    after = []
    for _ in range(2):
        rec.iterate(1, 0.5, 0.5)
        rec.image()
        replay()
        assert np.array_equal(_host_image(rec), want)
        assert np.array_equal(rec.image().cpu().numpy(), want)
        replay()
        rec.iterate(1, 0.5, 0.5)
        after.append(_host_image(rec))
    assert np.array_equal(after[0], after[1]) and not np.array_equal(after[0], want)
    rec.close()


@pytest.mark.parametrize("np_,J", [(32, 40), (64, 30), (128, 20)])
def test_replays_and_direct_calls_in_any_order(np_, J):
    """Whether a call finds the readout image of the state or gathers it is
    decided where the call runs: recorded and direct iterations on both sides of
    rho = 1/2 and recorded and direct states in a random order, every one of
    which begins and ends with rho = 1/2, against the direct calls alone."""
    import torch

    from paper_2111_14240_gb300 import pmace as pm
    rec, ref = _job(np_, J), _job(np_, J)
    state = []
    for r in (rec, ref):
        r.iterate(12, 0.5, 0.5)
        q = torch.empty((J, np_, np_, 2), device="cuda")
        xb = torch.empty((r.n1, r.n2, 2), device="cuda")
        state.append((q, xb, pm.pmace_get_state(r.h, q, xb)))

    def through_small_rho(r):
        r.iterate(1, 0.5, 0.3)
        r.iterate(1, 0.5, 0.5)

    calls = [lambda r, k: r.iterate(1, 0.5, 0.5), lambda r, k: r.iterate(3, 0.5, 0.5),
             lambda r, k: through_small_rho(r), lambda r, k: pm.pmace_set_state(r.h, *state[k])]
    replays = [_captured(lambda c=c: c(rec, 0)) for c in calls]
    calls.append(lambda r, k: r.iterate(11, 0.5, 0.5))   # replays a graph of the library's own: not recorded
    rng = np.random.Generator(np.random.PCG64(np_))
    for step in range(40):
        i = int(rng.integers(len(calls)))
        if i < len(replays) and rng.random() < 0.7:
            replays[i]()
        else:
            calls[i](rec, 0)
        calls[i](ref, 1)
        if rng.random() < 0.5:
            assert np.array_equal(_host_image(rec), ref.image().cpu().numpy()), step
    assert np.array_equal(rec.image().cpu().numpy(), ref.image().cpu().numpy())
    assert np.array_equal(rec.patches().cpu().numpy(), ref.patches().cpu().numpy())
    rec.close()
    ref.close()
