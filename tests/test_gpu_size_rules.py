"""Kernels and tile shapes chosen from a call's sizes, at the edges of each rule.

Neighbour list: batches up to 8192 atoms and bins are binned by one cluster launch and counts
up to 16384 are scanned by one block; larger ones take the general kernels.  GAP products:
tile widths follow the product's shape.  Results must not show which kernel ran.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import synth
from oracle import Params, basis, gap, neighbours, soap

pytestmark = pytest.mark.gpu

P4 = Params(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=3, l_max=1)


@pytest.fixture(scope="module", autouse=True)
def cuda_lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1905_02142_gb300 import build
    build.build()


def model_for(P, precision="mixed"):
    from paper_1905_02142_gb300.api import SoapGap
    return SoapGap.from_dict(dict(r_cut=P.r_cut, r_soft=P.r_soft, sigma_r0=P.sigma_r0, sigma_p0=P.sigma_p0,
                                  n_max=P.n_max, l_max=P.l_max, n_species=P.n_species), precision=precision)


def tiled(n_atoms):
    """n_atoms in copies of one 16-atom box and one box of the remainder, with the pair list
    made from the oracle's lists of the two."""
    boxes = [synth.random_box(16, side=6.5, dmin=1.0, seed=61, shear=0.2)] * (n_atoms // 16)
    if n_atoms % 16:
        boxes.append(synth.random_box(n_atoms % 16, side=5.1, dmin=1.0, seed=62))
    one = {id(b): neighbours.batch_pairs(synth.concat([b]), P4.r_cut) for b in boxes}
    i, j, s, off = [], [], [], 0
    for b in boxes:
        p = one[id(b)]
        i.append(p["i"] + off)
        j.append(p["j"] + off)
        s.append(p["shift"])
        off += b.n_atoms
    return synth.concat(boxes), np.concatenate(i), np.concatenate(j), np.concatenate(s)


@pytest.mark.parametrize("n_atoms", [1, 31, 33, 8191, 8192, 8193, 16384, 16385])
def test_pair_list_at_the_edges_of_the_small_kernels(n_atoms):
    from paper_1905_02142_gb300.api import Structures
    batch, i, j, s = tiled(n_atoms)
    m = model_for(P4)
    m.compute(Structures.from_batch(batch), desc=True)
    gi, gj, gs = m.pairs()
    assert np.array_equal(gi, i) and np.array_equal(gj, j) and np.array_equal(gs, s)


def test_pair_list_of_a_thin_cell_with_many_runs():
    """A cell far thinner than the cutoff: hundreds of (column, image) runs per atom, a few
    candidates each, so the runs are walked in several groups of 32."""
    from paper_1905_02142_gb300.api import Structures
    pos = np.array([[0.1, 0.1, 0.2], [0.7, 0.5, 1.9], [0.3, 0.2, 5.0]])
    cell = np.array([[0.9, 0.0, 0.0], [0.2, 1.3, 0.0], [0.0, 0.3, 7.0]])
    batch = synth.concat([synth.Structure(pos=pos, cell=cell, species=np.zeros(3, np.int32))])
    ref = neighbours.batch_pairs(batch, P4.r_cut)
    # the list names images of the atoms mapped into the cell (the third lies outside it in y)
    n = np.floor(pos @ np.linalg.inv(cell)).astype(np.int64)
    assert n.any()
    shift = ref["shift"] + n[ref["j"]] - n[ref["i"]]
    order = np.lexsort((shift[:, 2], shift[:, 1], shift[:, 0], ref["j"], ref["i"]))
    m = model_for(P4)
    m.compute(Structures.from_batch(batch), desc=True)
    gi, gj, gs = m.pairs()
    assert np.array_equal(gi, ref["i"][order]) and np.array_equal(gj, ref["j"][order])
    assert np.array_equal(gs, shift[order])


@pytest.mark.parametrize("sweep", [0, 1, 2])
def test_pair_list_of_every_bin_width(sweep):
    """The sweep by atom takes bins half the cutoff wide where a structure has an atom per such
    bin, the sweep by bin never does: cells around every multiple of half the cutoff, dense and
    sparse, sheared and elongated, in one batch."""
    from paper_1905_02142_gb300.api import Structures
    rc = P4.r_cut
    boxes = [synth.random_box(n, side=f * rc, dmin=0.2, seed=70 + k, shear=shear)
             for k, (n, f, shear) in enumerate([(4, 0.45, 0.0), (4, 0.5, 0.0), (5, 0.99, 0.2), (7, 1.0, 0.0),
                                                (8, 1.0, 0.0), (27, 1.5, 0.0), (26, 1.5, 0.0), (64, 2.0, 0.3),
                                                (130, 2.6, 0.0), (3, 2.6, 0.3), (40, 3.0, 0.0)])]
    rng = np.random.default_rng(71)
    long_cell = np.diag([2.1, 2.1, 60.0])
    boxes.append(synth.Structure(pos=rng.random((40, 3)) @ long_cell, cell=long_cell, species=np.zeros(40, np.int32)))
    batch = synth.concat(boxes)
    ref = neighbours.batch_pairs(batch, rc)
    m = model_for(P4)
    s = Structures.from_batch(batch)
    m.compute(s, desc=True)
    m.set_plan(s, {"adjoint_warps": 0, "gap_forward": 0, "gap_backward": 0, "neighbour_sweep": sweep, "pair_forward": 0})
    m.compute(s, desc=True)
    gi, gj, gs = m.pairs()
    assert np.array_equal(gi, ref["i"]) and np.array_equal(gj, ref["j"]) and np.array_equal(gs, ref["shift"])


@pytest.mark.parametrize("n,m_sparse", [(1, 1), (129, 33), (1000, 500), (4100, 260), (20001, 1030)])
def test_kernel_rows_of_every_tile_width(n, m_sparse):
    """Kernel rows of random unit descriptors against FP64 torch: both sides of the tile rule,
    ragged rows and columns, row strides that are not a multiple of 4 floats.  The split FP16
    products carry ~2^-21 of |u_i . u_s| <= 1 and the FP32 sum of three terms 3 * 2^-24, each
    times zeta = 3: below 3 * (2^-21 + 2^-22) = 2.2e-6."""
    rng = np.random.default_rng(n)
    m = model_for(Params(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=5, l_max=3))
    q = np.abs(rng.normal(1.0, 0.2, (n + m_sparse, m.dim)))
    q = (q / np.linalg.norm(q, axis=1, keepdims=True)).astype(np.float32)
    m.set_model(q[n:].astype(np.float64), rng.normal(0, 0.1, m_sparse), 3.0)
    k = m.kernel_rows(torch.as_tensor(q[:n], device="cuda"))
    ref = (torch.as_tensor(q[:n]).double() @ torch.as_tensor(q[n:]).double().T) ** 3
    assert float((k.cpu().double() - ref).abs().max()) < 2.2e-6


@pytest.mark.parametrize("n_max,l_max,alpha_r", [(6, 8, 0.0), (6, 12, 0.0), (5, 8, 0.1), (4, 0, 0.0)])
def test_fp64_distance_factors_of_every_branch(n_max, l_max, alpha_r):
    """FP64 dimers at distances on both sides of each branch of the distance factors: z = (r /
    sigma)^2 below and above 1e-3 (series) and 30 (upward recursion), r in the buffer zone and
    next to the cutoff; the hoisted analytic form (n, l <= 8, alpha_r = 0) and the general one.
    Bars as the other FP64 parity tests: 1e-11 or 4 eps sqrt(cond S) on p, 1e-9 or twice that
    scale on forces."""
    from paper_1905_02142_gb300.api import SoapGap, Structures
    P = Params(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, alpha_r=alpha_r, n_max=n_max, l_max=l_max)
    dist = [0.01, 0.0158, 0.0159, 0.5, 1.3, 2.7386, 2.7387, 3.4999, 3.5001, 3.99]
    u = np.array([0.48, -0.6, 0.64])
    batch = synth.concat([synth.Structure(pos=np.array([[5.0, 5.0, 5.0], [5.0, 5.0, 5.0] + r * u]),
                                          cell=np.eye(3) * 12.0, species=np.zeros(2, np.int32)) for r in dist])
    W = basis.orthonormaliser(P.n_max, P.r_cut, P.sigma_r0)
    ref = soap.descriptors(batch, P, W=W)
    qs = ref["q"].numpy()[[6, 8, 19]] + 0.01
    al = np.array([0.3, -0.2, 0.5])
    full = gap.evaluate(batch, P, qs, al, 3.0, W=W, virial=False)
    m = SoapGap(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, alpha_r=alpha_r, n_max=n_max, l_max=l_max,
                precision="fp64")
    m.set_model(qs, al, 3.0)
    out = m.compute(Structures.from_batch(batch), desc=True, energy=True, forces=True)
    p = (out["q"] * out["pnorm"][:, None]).cpu().numpy()
    p_ref = (ref["q"] * ref["pnorm"][:, None]).numpy()
    r = np.finfo(float).eps * np.sqrt(np.linalg.cond(W @ W))   # cond(S) = cond(W)^2
    assert np.max(np.linalg.norm(p - p_ref, axis=1) / np.linalg.norm(p_ref, axis=1)) < max(1e-11, 4 * r)
    f, f_ref = out["forces"].cpu().numpy(), full["forces"]
    assert np.linalg.norm(f - f_ref) / np.linalg.norm(f_ref) < max(1e-9, 2 * r)


@pytest.mark.parametrize("n_max,l_max,nsp,atoms", [(3, 0, 1, 20), (5, 0, 1, 20), (5, 8, 1, 20), (4, 12, 1, 20),
                                                   (12, 7, 1, 20), (9, 10, 1, 20), (3, 3, 3, 20), (8, 8, 2, 20),
                                                   (8, 8, 1, 520), (8, 10, 1, 520)])
def test_force_rows_of_every_descriptor_shape(n_max, l_max, nsp, atoms):
    """Force rows of the fitting matrices, mixed against FP64: descriptors whose length leaves 6
    or 7 entries in the last 8 (the two carried terms then lie in two pieces), runs of l shorter
    and longer than 8, one and several groups of 8 channels; 520 atoms have enough columns for
    the stationary-tile GEMM, with 6 and 7 blocks of K.  Bar: 1e-3 RMS, the mixed path's for
    forces."""
    from paper_1905_02142_gb300.api import Structures
    probs = None if nsp == 1 else [1.0 / nsp] * nsp
    P = Params(r_cut=5.0, r_soft=4.5, sigma_r0=0.5, sigma_p0=0.5, n_max=n_max, l_max=l_max, n_species=nsp)
    batch = synth.concat([synth.random_box(atoms, density=0.15, dmin=1.1, seed=71, species_probs=probs)])
    sb = synth.concat([synth.random_box(140, density=0.15, dmin=1.1, seed=72, species_probs=probs)])
    ref = model_for(P, "fp64")
    qs = ref.compute(Structures.from_batch(sb), desc=True)["q"].cpu().numpy()[:130]
    rows = {}
    for precision in ("fp64", "mixed"):
        m = model_for(P, precision)
        m.set_model(qs, np.ones(len(qs)), 2.0)
        rows[precision] = m.design(Structures.from_batch(batch), k_struct=True, dk=True)["dk"].double().cpu()
    assert float((rows["mixed"] - rows["fp64"]).norm() / rows["fp64"].norm()) < 1e-3


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_calls_that_run_ahead_of_their_pair_count(precision):
    """Calls after the first on a batch of the same shape do not wait for their pair count.
    Whatever the next configuration needs (as many pairs, a cluster that outgrows the slots, more
    pairs than the buffers hold, another problem class, few pairs, then the first again), its
    results and pair list are those of a fresh handle, bit for bit; a position that is not finite
    is reported as before and does not disturb the next call."""
    from paper_1905_02142_gb300 import _lib
    from paper_1905_02142_gb300.api import SoapGapError, Structures
    P = Params(r_cut=4.5, r_soft=4.0, sigma_r0=0.5, sigma_p0=0.5, n_max=4, l_max=3)
    base = synth.concat([synth.random_box(216, density=0.10, dmin=1.1, seed=81)])
    side = float(base.cell[0, 0, 0])
    sb = synth.concat([synth.random_box(30, density=0.10, dmin=1.1, seed=82)])
    qs = model_for(P, "fp64").compute(Structures.from_batch(sb), desc=True)["q"].cpu().numpy()
    al = np.random.default_rng(83).normal(0, 0.1, len(qs))

    def model():
        m = model_for(P, precision)
        m.set_model(qs, al, 2.0)
        return m

    def at(scale, cell_scale=1.0):
        return synth.Batch(pos=base.pos * scale, cell=base.cell * cell_scale, species=base.species,
                           atom_offs=base.atom_offs)
    want = dict(energy=True, forces=True, virial=True)
    m = model()
    m.compute(Structures.from_batch(at(1.0)), **want)
    shifted = at(1.0)
    shifted.pos[:] += 0.37 * side
    for k, b in enumerate([shifted, at(0.6), at(0.45), at(0.8, 0.8), at(3.0, 3.0), at(1.0), at(1.0)]):
        out = m.compute(Structures.from_batch(b), **want)
        got = m.pairs()
        fresh = model()
        ref = fresh.compute(Structures.from_batch(b), **want)
        for name in ref:
            assert torch.equal(out[name], ref[name]), (k, name)
        for x, y in zip(got, fresh.pairs()):
            assert np.array_equal(x, y), k
    bad = at(1.0)
    bad.pos[5, 1] = np.nan
    with pytest.raises(SoapGapError) as err:
        m.compute(Structures.from_batch(bad), **want)
    assert err.value.code == _lib.E_INVALID_ARG and "not finite" in str(err.value)
    again = m.compute(Structures.from_batch(at(1.0)), **want)
    for name in ref:
        assert torch.equal(again[name], ref[name]), name


@pytest.mark.parametrize("n_max,l_max", [(4, 6), (6, 3), (5, 6), (8, 4), (8, 5), (3, 8), (6, 7), (10, 4), (10, 6),
                                         (9, 8), (4, 10), (7, 9), (12, 5), (12, 8), (11, 10), (3, 11), (6, 12), (9, 12)])
def test_forward_kernel_of_every_evaluated_size(n_max, l_max):
    """The forward pair kernel evaluates n_max and l_max rounded up to even (at least 4) within
    the basis class: every such pair of bounds, both precisions, against the oracle.  Bars: 1e-5
    on p mixed, 1e-11 or 4 eps sqrt(cond S) in FP64."""
    from paper_1905_02142_gb300.api import Structures
    P = Params(r_cut=4.0, r_soft=3.5, sigma_r0=0.5, sigma_p0=0.5, n_max=n_max, l_max=l_max, n_species=2)
    batch = synth.concat([synth.random_box(24, density=0.12, dmin=1.1, seed=91, species_probs=[0.6, 0.4])])
    ref = soap.descriptors(batch, P)
    p_ref = (ref["q"] * ref["pnorm"][:, None]).numpy()
    r = np.finfo(float).eps * np.sqrt(np.linalg.cond(basis.overlap_matrix(n_max, 4.0, 0.5)))
    for precision, bar in (("mixed", 1e-5), ("fp64", max(1e-11, 4 * r))):
        out = model_for(P, precision).compute(Structures.from_batch(batch), desc=True)
        p = (out["q"].double() * out["pnorm"].double()[:, None]).cpu().numpy()
        assert np.max(np.linalg.norm(p - p_ref, axis=1) / np.linalg.norm(p_ref, axis=1)) < bar, precision
