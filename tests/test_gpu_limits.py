"""Models and calls past the usual sizes, against the FP64 oracle.

Bounds, those of the parity tests: FP32 forces within 1e-4 of their RMS, energies within
1e-3 kcal/mol and within 1e-4 of sum_i |E_i|; BF16 forces within 2e-2 of their RMS (2^-9
relative per operand); gradients of the loss within 1e-3 of their norm and largest element.
"""
import numpy as np
import pytest

import oracle
import synth
from tests._common import to_cuda
from tests.test_gpu_shapes import check, close, model

gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


# the last backward layer sums over all members' first hidden layers: 32 slices of 64
# columns fill a mask word, 33, 35 and 45 are past it
@gpu
@pytest.mark.parametrize("precision", ["fp32_split", "bf16", "fp32_simt"])
@pytest.mark.parametrize("ensemble,hidden", [(8, (256, 64, 32)), (11, (192, 48, 16)), (7, (320, 64, 48)), (9, (320, 32, 32))])
def test_first_layers_of_all_members_past_2048_columns(torch_cuda, precision, ensemble, hidden):
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4", hidden, ensemble)
    pot, orc = Potential(spec, w, precision=precision), oracle.Model(spec, w)
    systems = [synth.water_box(60, 12.2, 4, seed=61)] + list(synth.workload("molecules64")[0][:2])
    for sparse in (False, True):
        pot.set_sparse_rows(sparse)
        check(pot, orc, systems, precision)


# Sections of 0 .. 0.7 rad and two neighbours on opposite sides of a centre: 1 + cos(theta -
# theta_z) is exactly 0 in the first section (the distance 2 and its reciprocal are exact) and
# below 0.24 in the others, whose 32nd powers vanish.  (The two are farther apart than the
# angular cutoff: seen from one of them the others would lie on one side, where the energy has
# a cusp.)  The oracle, which divides by sin(theta), has the pair 1e-7 A off the line.
def collinear():
    spec, w = model("ani4", shf_z=tuple(0.1 * z for z in range(8)))
    x = np.array([[0, 0, 0], [0, 0, 2], [0, 0, -2], [1.25, 0.5, 0.25], [-1.5, 0.75, 0.5]], np.float32)
    s = synth.systems.System("collinear", x, np.array([1, 3, 3, 0, 0], np.uint8))
    off = x.astype(np.float64)
    off[1, 0] += 1e-7
    return spec, w, s, off


@gpu
@pytest.mark.parametrize("precision", ["fp32", "fp32_simt", "bf16"])
def test_a_section_opposite_to_a_collinear_pair(torch_cuda, precision):
    from paper_2207_14276_gb300 import Potential
    spec, w, s, off = collinear()
    ref = oracle.Model(spec, w).energy_forces(off, s.species)
    assert np.isfinite(ref["forces"]).all()
    pot = Potential(spec, w, precision=precision)
    far = synth.water_box(300, 20.5, 7, seed=41)   # beside it, centres have a warp each
    for systems in ([s], [s, far]):
        o = pot.energy_forces_batch([to_cuda(q) for q in systems])[0]
        close(o, ref, precision)


@gpu
def test_gradients_with_a_section_opposite_to_a_collinear_pair(torch_cuda):
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    spec, w, s, off = collinear()
    pot, orc = Potential(spec, w), oracle.Model(spec, w)
    v = np.random.Generator(np.random.PCG64(12)).normal(size=(s.n_atoms, 3))
    _, _, gx, gw = pot.force_vjp_batch([to_cuda(s)], [0.0], [torch.from_numpy(v).float().cuda()])
    _, _, gx_ref, gw_ref = orc.force_matching(off, s.species, v.astype(np.float32))
    for got, ref in ((gx[0], gx_ref), (gw, gw_ref)):
        assert np.isfinite(ref).all()
        d = got.cpu().numpy().astype(np.float64) - ref
        assert np.linalg.norm(d) <= 1e-3 * np.linalg.norm(ref)
        assert np.abs(d).max() <= 1e-3 * np.abs(ref).max()


# the network gradient read back after a call for energies alone, which forms none: the read
# runs the ensemble's backward (1e-4 of the norm: the parity test's bound of an element)
@gpu
@pytest.mark.parametrize("sparse", [True, False])
def test_gradient_rows_after_an_energy_only_call(torch_cuda, sparse):
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4", ensemble=3)
    pot, orc = Potential(spec, w, precision="fp32_simt"), oracle.Model(spec, w)
    pot.set_sparse_rows(sparse)
    s = synth.water_box(60, 12.2, 4, seed=61)
    ref = orc.energy_forces(s.coords, s.species, s.box, want_dEdG=True)["dEdG"]
    other = to_cuda(synth.water_box(60, 12.2, 4, seed=62))
    d = to_cuda(s)

    def read():
        g = pot.debug_rows(1, s.n_atoms).cpu().numpy()
        assert np.linalg.norm(g - ref) <= 1e-4 * np.linalg.norm(ref)

    for _ in range(3):   # eager, captured, replayed
        pot.energy_forces_batch([d], forces=False)
        read()
        read()
    pot.energy_forces_batch([other])
    pot.energy_forces_batch([d])
    read()
    pot.energy_forces_batch([other])
    pot.energy_forces_batch([d], forces=False)
    read()


# shapes that take turns on a handle: a graph that another shape's replaces after a call or two
# costs more than it saves.  Captures end after a few turns, and a shape that stays gets its graph
@gpu
@pytest.mark.parametrize("turn", ["AB", "AAB", "AABB", "AAABBB", "AABBCC"])
def test_shapes_that_take_turns_are_not_captured_each_turn(torch_cuda, turn):
    from paper_2207_14276_gb300 import Potential, _lib
    spec, w = model("ani4")
    pot, orc = Potential(spec, w), oracle.Model(spec, w)
    systems = dict(zip("ABC", synth.workload("molecules64")[0][:3]))
    dev = {k: to_cuda(s) for k, s in systems.items()}
    refs = {k: orc.energy_forces(s.coords, s.species) for k, s in systems.items()}

    def captures():
        return _lib.lib().nnp_debug_graph_captures(pot._h)

    def call(k):
        E, F = pot.energy_forces(dev[k]["coords"], dev[k]["species"])
        return {"energy": E, "forces": F}

    for _ in range(12):
        for k in turn:
            call(k)
    settled = captures()
    assert settled <= 6   # the wait doubles from 2 to 64
    for _ in range(12):
        for k in turn:
            close(call(k), refs[k], "fp32")
    assert captures() == settled
    for k in "CBA":
        for _ in range(70):
            call(k)
        n = captures()
        close(call(k), refs[k], "fp32")
        assert captures() == n and n >= settled
    assert captures() > settled


# rows are grouped by their live slices past 32,768 atoms, or where slices times networks exceed
# 8: the same results as whole rows to the last bits of sums of products (1e-5 of the norm), with
# lists kept between calls too
@gpu
@pytest.mark.parametrize("kind,ensemble,n_mol", [("ani4", 1, 10922), ("ani4", 1, 10923), ("ani4", 2, 500)])
def test_rows_grouped_or_not(torch_cuda, kind, ensemble, n_mol):
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    spec, w = model(kind, ensemble=ensemble)
    pot = Potential(spec, w)
    edge = 44.77 * (n_mol / 3000) ** (1 / 3)
    s = synth.water_box(n_mol, edge, int(np.ceil(n_mol ** (1 / 3))), seed=71)
    d = to_cuda(s)
    pot.set_sparse_rows(False)
    E0, F0 = pot.energy_forces(d["coords"], d["species"], d["box"])
    pot.set_sparse_rows(True)
    for skin in (0.0, 0.5):
        pot.set_skin(skin)
        for _ in range(3):
            E, F = pot.energy_forces(d["coords"], d["species"], d["box"])
            assert float((F - F0).norm()) <= 1e-5 * float(F0.norm())
            assert abs(float(E[0] - E0[0])) <= 1e-6 * abs(float(E0[0])) + 1e-6 * s.n_atoms ** 0.5
    pot.set_skin(0.0)
