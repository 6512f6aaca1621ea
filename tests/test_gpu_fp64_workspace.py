"""FP64 path: the workspace of distance factors serves asynchronous calls and captured graphs
whatever synchronous calls came between."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02142_gb300 import build
    build.build()


def setup(n_max):
    from paper_1905_02142_gb300.api import SoapGap, Structures
    model = SoapGap(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=n_max, l_max=3, precision="fp64")
    rng = np.random.default_rng(5)
    q = np.abs(rng.normal(size=(20, model.dim)))
    model.set_model(q / np.linalg.norm(q, axis=1, keepdims=True), rng.normal(0, 0.1, 20), 2.0)
    a, b = (Structures.from_batch(synth.concat([synth.random_box(n, density=0.1, dmin=1.1, seed=n)]))
            for n in (200, 2000))
    return model, a, b


@pytest.mark.parametrize("n_max", [4, 9])   # one pass with derivatives, and two passes
def test_asynchronous_call_after_descriptors_of_a_larger_batch(n_max):
    model, a, b = setup(n_max)
    ref = {k: v.clone() for k, v in model.compute(a, energy=True, forces=True).items()}
    model.compute(b, desc=True)              # grows the pair buffers
    out = model.compute(a, energy=True, forces=True, asynchronous=True)
    model.sync_status()
    for k in ref:
        assert torch.equal(out[k], ref[k]), k


@pytest.mark.parametrize("n_max", [4, 9])
def test_captured_energies_after_forces_of_the_same_batch(n_max):
    from paper_1905_02142_gb300.api import CapturedEvaluation
    model, a, _ = setup(n_max)
    ref = {k: v.clone() for k, v in model.compute(a, energy=True).items()}
    cap = CapturedEvaluation(model, a, energy=True)
    model.compute(a, energy=True, forces=True)
    out = cap.replay()
    model.sync_status()
    for k in ref:
        assert torch.equal(out[k], ref[k]), k
