"""The largest descriptors that a kernel's shared memory takes."""
import numpy as np
import pytest
import torch

import synth
from oracle import Params, basis, soap

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02142_gb300 import build
    build.build()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_descriptors_of_six_species_against_oracle(precision):
    """n_max = 9, l_max = 11 and six species: one FP64 atom's rows and descriptor fill 204,768 bytes,
    205,632 with the rows' padding.  Bars: 1e-5 on p mixed, 1e-11 or 4 eps sqrt(cond S) in FP64."""
    from paper_1905_02142_gb300.api import SoapGap, Structures
    P = Params(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=9, l_max=11, n_species=6)
    batch = synth.concat([synth.random_box(9, density=0.08, dmin=1.1, seed=95, species_probs=[1 / 6] * 6)])
    ref = soap.descriptors(batch, P)
    p_ref = (ref["q"] * ref["pnorm"][:, None]).numpy()
    r = np.finfo(float).eps * np.sqrt(np.linalg.cond(basis.overlap_matrix(9, 4.0, 0.5)))
    bar = 1e-5 if precision == "mixed" else max(1e-11, 4 * r)
    m = SoapGap(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=9, l_max=11, n_species=6, precision=precision)
    out = m.compute(Structures.from_batch(batch), desc=True)
    p = (out["q"].double() * out["pnorm"].double()[:, None]).cpu().numpy()
    assert np.max(np.linalg.norm(p - p_ref, axis=1) / np.linalg.norm(p_ref, axis=1)) < bar
