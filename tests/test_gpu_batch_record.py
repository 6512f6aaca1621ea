"""Asynchronous calls and graph replays read the batch's geometry when they run, from staging
that later calls on the handle use too: those calls must not change what they read."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

OUT = dict(energy=True, forces=True, virial=True)


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02142_gb300 import build
    build.build()


def make_model(n_max=4, l_max=4, m_sparse=64, r_cut=4.0):
    from paper_1905_02142_gb300.api import SoapGap
    model = SoapGap(r_cut=r_cut, r_soft=r_cut - 0.5, sigma_r0=0.5, sigma_p0=0.5, n_max=n_max, l_max=l_max,
                    precision="mixed")
    rng = np.random.default_rng(3)
    q = np.abs(rng.normal(size=(m_sparse, model.dim)))
    model.set_model(q / np.linalg.norm(q, axis=1, keepdims=True), synth.gap_weights(m_sparse, 4), 2.0)
    return model


def check_equal(out, ref):
    for k in ("e_struct", "forces", "e_atom"):
        assert torch.equal(out[k], ref[k]), k
    assert torch.allclose(out["virial"], ref["virial"], rtol=1e-12, atol=0)


def busy(ms):
    """About `ms` milliseconds of other work on the current stream."""
    torch.cuda._sleep(int(ms * 1.9e6))


def test_queued_calls_on_one_batch_keep_their_geometry():
    """Asynchronous calls queued behind other work, their geometry copies still pending while the
    later ones are set up, give the results of a synchronous call."""
    from paper_1905_02142_gb300.api import Structures
    batch = synth.batched_boxes(256, n_lo=1, n_hi=200, seed=21)
    model = make_model()
    s = Structures.from_batch(batch)
    ref = {k: v.clone() for k, v in model.compute(s, **OUT).items()}
    for _ in range(3):
        torch.cuda.synchronize()
        busy(20.0)
        outs = [model.compute(s, asynchronous=True, **OUT) for _ in range(12)]
        model.sync_status()
        for out in outs:
            check_equal(out, ref)


@pytest.mark.parametrize("captured,later", [(1, 2), (2, 1)])
@pytest.mark.parametrize("structures", [1, 12])
def test_replay_after_a_call_with_the_other_sweep(structures, captured, later):
    """A graph captured under one candidate sweep replays the same after synchronous calls on its
    batch that sweep the other way, by another plan for its problem class or because its pairs
    per atom moved it to a class with another plan.  (The capture sees the densest configuration:
    a synchronous call with more pairs than the buffers hold reallocates them.)"""
    from paper_1905_02142_gb300.api import CapturedEvaluation, Structures
    if structures == 1:
        batch = synth.concat([synth.random_box(3000, density=0.12, dmin=1.0, seed=22)])
    else:
        batch = synth.batched_boxes(structures, n_lo=20, n_hi=400, seed=23)
    model = make_model()
    s = Structures.from_batch(batch)
    loose = s.pos.clone()
    dense = loose * 0.85
    plan = {"adjoint_warps": 0, "gap_forward": 0, "gap_backward": 0, "pair_forward": 0}
    s.pos.copy_(dense)
    model.compute(s, **OUT)
    model.set_plan(s, dict(plan, neighbour_sweep=captured))
    ref = {k: v.clone() for k, v in model.compute(s, **OUT).items()}
    pairs = model.pair_count()
    cap = CapturedEvaluation(model, s, **OUT)
    check_equal(cap.replay(), ref)
    model.sync_status()
    # the other sweep in this class, and in the class of a looser configuration
    for at in (dense, loose):
        s.pos.copy_(at)
        model.compute(s, **OUT)
        model.set_plan(s, dict(plan, neighbour_sweep=later))
        for _ in range(2):   # the second call runs ahead of its pair count
            again = model.compute(s, **OUT)
        assert model.pair_count() <= pairs
        if at is dense:
            check_equal(again, ref)
        s.pos.copy_(dense)
        for _ in range(4):
            check_equal(cap.replay(), ref)
            model.sync_status()
