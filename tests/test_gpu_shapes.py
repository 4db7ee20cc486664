"""The kernels at the edges of the sizes they divide their work by, against the FP64
oracle: layer widths at and past the limits of the fused last-layer kernel, batches
around the size up to which a centre has a CTA of its own, centres around the neighbour
count that makes them dense, masked regions of a few rows, odd network widths and
exponents of the differentiation, and a call's graph under new buffers, other streams
and capture.

Bounds, those of the parity tests: FP32 forces within 1e-4 of their RMS, energies within
1e-3 kcal/mol and within 1e-4 of sum_i |E_i| (operands of 16 bits on the split path); BF16
forces within 2e-2 of their RMS (2^-9 relative per operand; its energies, whose error is a
bias per member that does not shrink where members cancel, are compared between two
kernels); gradients of the loss within 1e-3 of their norm and largest element.
"""
import dataclasses

import numpy as np
import pytest

import oracle
import synth
from tests._common import force_errors, to_cuda

gpu = pytest.mark.gpu
FP32 = ("fp32", "fp32_split", "fp32_simt")


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


def model(kind="ani4", hidden=None, ensemble=None, seed=1, **aev):
    spec = synth.model_spec(kind)
    if hidden:
        spec = dataclasses.replace(spec, widths=(spec.widths[0], *hidden, 1))
    if ensemble:
        spec = dataclasses.replace(spec, n_ensemble=ensemble)
    if aev:
        spec = dataclasses.replace(spec, aev=dataclasses.replace(spec.aev, **aev))
    return spec, synth.make_weights(spec, seed)


def close(out, ref, precision, mask=None):
    F = out["forces"].cpu().numpy()
    rms, _ = force_errors(F, ref["forces"])
    f_rms = float(np.sqrt(np.mean(ref["forces"] ** 2)))
    if precision in FP32:
        scale = float(np.abs(ref["atom_energies"]).sum())
        dE = abs(float(out["energy"].cpu()[0]) - ref["energy"])
        assert rms <= 1e-4 * f_rms + 1e-7
        assert dE <= min(1e-3, 1e-4 * scale + 1e-6)
    else:
        assert rms <= 2e-2 * f_rms + 1e-6
    if mask is not None:
        assert np.all(F[mask == 0] == 0.0)


def check(pot, orc, systems, precision, **kw):
    outs = pot.energy_forces_batch([to_cuda(s) for s in systems], **kw)
    for s, o in zip(systems, outs):
        ref = orc.energy_forces(s.coords, s.species, s.box, s.mask)
        close(o, ref, precision, s.mask)
        if kw.get("virial") and s.box is not None:
            np.testing.assert_allclose(o["virial"].cpu().numpy().reshape(3, 3), ref["virial"],
                                       atol=1e-4 * np.abs(ref["virial"]).max() + 1e-6)
    return outs


# 512 tensor-memory columns hold two z3 accumulators (h3 up to a multiple of 32) and one
# delta2: (256, 128) fills them, (208, 160) and (176, 176) do not fit; 192 is the widest
# h3; 80 and 48 leave partial K slices and 64-column blocks
@gpu
@pytest.mark.parametrize("precision", ["fp32_split", "bf16"])
@pytest.mark.parametrize("hidden,ensemble", [
    ((64, 16, 16), 1), ((96, 64, 64), 2), ((48, 80, 48), 3), ((256, 256, 128), 1), ((256, 208, 160), 2),
    ((192, 176, 176), 1), ((64, 48, 192), 1), ((256, 192, 160), 2)])
def test_last_layer_widths(torch_cuda, precision, hidden, ensemble):
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4", hidden, ensemble)
    pot, orc = Potential(spec, w, precision=precision), oracle.Model(spec, w)
    systems = [synth.water_box(300, 20.5, 7, seed=41)] + list(synth.workload("molecules64")[0][:3])
    outs = check(pot, orc, systems, precision)
    alone = pot.energy_forces_batch([to_cuda(s) for s in systems], forces=False)
    for a, o, s in zip(alone, outs, systems):   # the energies alone, by L3's layer GEMM
        scale = np.abs(orc.energy_forces(s.coords, s.species, s.box)["atom_energies"]).sum()
        assert abs(float(a["energy"].cpu()[0]) - float(o["energy"].cpu()[0])) <= 1e-5 * scale + 1e-6


@gpu
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_several_tiles_per_cta(torch_cuda, precision):
    # 46 row tiles x 8 members: two to three tiles per CTA of the fused last-layer kernel
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani7x8")
    pot, orc = Potential(spec, w, precision=precision), oracle.Model(spec, w)
    s = synth.solvated_solute(1800, 60, 39.0, seed=6)
    check(pot, orc, [s], precision)


@gpu
@pytest.mark.parametrize("n", [1, 2, 31, 33, 607, 608, 609])
def test_masked_region_sizes(torch_cuda, n):
    # the centres of a mask around the count that gives each a CTA, and few row tiles
    # in launches sized for all atoms
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4")
    s = synth.water_box(900, 30.0, 10, seed=3)
    mask = np.zeros(s.n_atoms, np.uint8)
    mask[np.random.Generator(np.random.PCG64(n)).permutation(s.n_atoms)[:n]] = 1
    s = dataclasses.replace(s, mask=mask)
    check(Potential(spec, w), oracle.Model(spec, w), [s], "fp32")


@gpu
@pytest.mark.parametrize("precision", ["fp32", "bf16"])
def test_masked_solute_of_a_large_box(torch_cuda, precision):
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani7x8")
    s = synth.solvated_solute(1500, 50, 37.0, seed=9, mask_solute=True)
    check(Potential(spec, w, precision=precision), oracle.Model(spec, w), [s], precision)


def cluster(na, seed):
    """One centre with exactly na neighbours within 3.5 A, at least 1.1 A apart."""
    rng = np.random.Generator(np.random.PCG64(seed))
    x = [np.zeros(3)]
    while len(x) < na + 1:
        v = rng.normal(size=3)
        v *= rng.uniform(1.2, 3.4) / np.linalg.norm(v)
        if min(np.linalg.norm(v - y) for y in x) > (1.1 if len(x) < 34 else 0.9):
            x.append(v)
    sp = (np.arange(na + 1) % 4).astype(np.uint8)
    return synth.systems.System("cluster", np.array(x, np.float32), sp)


@gpu
@pytest.mark.parametrize("precision", ["fp32", "fp32_simt"])
@pytest.mark.parametrize("na", [31, 32, 33, 64])
def test_dense_centre_threshold(torch_cuda, precision, na):
    # beside 900 water atoms, so that the other centres have a warp each; with virials
    # of two boxes and repeated calls (the second replays the first's graph)
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4")
    pot, orc = Potential(spec, w, precision=precision), oracle.Model(spec, w)
    systems = [cluster(na, na), synth.water_box(300, 20.5, 7, seed=41), synth.water_box(100, 14.5, 5, seed=61)]
    for _ in range(2):
        check(pot, orc, systems, precision, virial=True)


@gpu
@pytest.mark.parametrize("ensemble,hidden", [(1, (160, 128, 96)), (3, (48, 80, 16)), (8, (64, 48, 32))])
def test_sparse_rows_of_fp32_networks(torch_cuda, ensemble, hidden):
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani7", hidden, ensemble)
    pot, orc = Potential(spec, w, precision="fp32_simt"), oracle.Model(spec, w)
    systems = [synth.solvated_solute(200, 40, 20.0, seed=6)]
    for sparse in (False, True):
        pot.set_sparse_rows(sparse)
        check(pot, orc, systems, "fp32_simt")


@gpu
@pytest.mark.parametrize("kind,hidden,ensemble,aev", [
    ("ani7", None, 1, {}), ("ani7", (48, 80, 32), 3, {}), ("ani4", (64, 48, 16), 2, {"cos_scale": 0.95}),
    ("ani4", None, 1, {"zeta": 14.0})])
def test_force_matching_shapes(torch_cuda, kind, hidden, ensemble, aev):
    # two molecules and a box with a mask, dL/dE and dL/dF at once
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    spec, w = model(kind, hidden, ensemble, **aev)
    pot, orc = Potential(spec, w), oracle.Model(spec, w)
    rng = np.random.Generator(np.random.PCG64(12))
    box = synth.water_box(40, 12.0, 4, seed=5)
    mask = np.zeros(box.n_atoms, np.uint8)
    mask[:75] = 1
    systems = list(synth.workload("molecules64")[0][:2]) + [dataclasses.replace(box, mask=mask)]
    v = [rng.normal(size=(s.n_atoms, 3)) for s in systems]
    c = [0.5, -1.0, 2.0]
    _, _, gx, gw = pot.force_vjp_batch([to_cuda(s) for s in systems], c,
                                       [torch.from_numpy(u).float().cuda() for u in v])
    gw_ref = np.zeros(w.size)
    for k, s in enumerate(systems):
        r = orc.energy_forces(s.coords, s.species, s.box, s.mask, want_dEdW=True)
        vv = v[k] if s.mask is None else v[k] * s.mask[:, None]
        _, _, gxk, gwk = orc.force_matching(s.coords, s.species, vv, s.box, s.mask)
        gw_ref += gwk + c[k] * r["dEdW"]
        ref = gxk - c[k] * r["forces"]
        d = gx[k].cpu().numpy().astype(np.float64) - ref
        assert np.linalg.norm(d) <= 1e-3 * np.linalg.norm(ref)
        assert np.abs(d).max() <= 1e-3 * np.abs(ref).max()
    d = gw.cpu().numpy().astype(np.float64) - gw_ref
    assert np.linalg.norm(d) <= 1e-3 * np.linalg.norm(gw_ref)
    assert np.abs(d).max() <= 1e-3 * np.abs(gw_ref).max()


@gpu
@pytest.mark.parametrize("n_mol", [40, 300])
def test_one_graph_for_new_buffers_streams_and_capture(torch_cuda, n_mol):
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    spec, w = model("ani4")
    pot, orc = Potential(spec, w), oracle.Model(spec, w)
    edge, side = (12.0, 4) if n_mol == 40 else (20.5, 7)
    boxes = [synth.water_box(n_mol, edge, side, seed=70 + k) for k in range(4)]
    streams = [None, None, torch.cuda.Stream(), None]
    for s, st in zip(boxes, streams):   # fresh inputs and outputs on every call
        with torch.cuda.stream(st or torch.cuda.current_stream()):
            check(pot, orc, [s], "fp32")
    # a capture of the caller's own, replayed with other coordinates in place
    d = to_cuda(boxes[0])
    E = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.zeros((boxes[0].n_atoms, 3), dtype=torch.float32, device="cuda")
    side_stream = torch.cuda.Stream()
    side_stream.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side_stream):
        pot.energy_forces_into(d["coords"], d["species"], d["box"], None, E, F)
    for s in (boxes[1], boxes[0]):
        d["coords"].copy_(torch.from_numpy(s.coords))
        d["species"].copy_(torch.from_numpy(s.species))
        g.replay()
        torch.cuda.synchronize()
        pot.sync_status()
        close({"energy": E, "forces": F}, orc.energy_forces(s.coords, s.species, s.box), "fp32")
    check(pot, orc, [boxes[3]], "fp32")


@gpu
def test_batch_sizes_as_torch_split_takes_them(torch_cuda):
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    from paper_2207_14276_gb300.autograd import NNPBatchFunction
    spec, w = model("ani4")
    pot = Potential(spec, w)
    s = to_cuda(synth.workload("gas24")[0][0])
    x, wt = s["coords"].repeat(3, 1)[:60].contiguous(), torch.from_numpy(w).cuda()
    sp = s["species"].repeat(3)[:60].contiguous()
    out = [NNPBatchFunction.apply(x, wt, pot, sp, sizes) for sizes in (24, [24, 24, 12], (24, 24, 12))]
    for E, F in out[1:]:
        torch.testing.assert_close(E, out[0][0], rtol=1e-6, atol=1e-6)
        torch.testing.assert_close(F, out[0][1], rtol=1e-5, atol=1e-5)
    with pytest.raises(TypeError):
        NNPBatchFunction.apply(x, wt, pot, sp, [24.0, 24.0, 12.0])
    with pytest.raises(RuntimeError):
        NNPBatchFunction.apply(x, wt, pot, sp, [24, 24])


# a budget of what lists, rows and activations alone take has room for the call: the row
# groups and output parts lie in the FP32 rows, or the FMA paths run without masks
@gpu
@pytest.mark.parametrize("kind,precision,ensemble", [
    ("ani7", "fp32", 1), ("ani7x8", "bf16", 8), ("ani7x8", "fp32_simt", 8), ("ani7", "fp32_simt", 1)])
def test_a_budget_of_the_arena_without_extras(torch_cuda, kind, precision, ensemble):
    from paper_2207_14276_gb300 import Potential
    from paper_2207_14276_gb300._lib import NNPError
    spec, w = model(kind)
    systems = [synth.solvated_solute(400, 60, 24.0, seed=6)]
    room = (systems[0].n_atoms, 1, 288, 96)
    with pytest.raises(NNPError) as e:
        Potential(spec, w, precision=precision, hbm_budget=1).reserve(*room)
    need = int(str(e.value).split("work arena of ")[1].split()[0])
    pot, orc = Potential(spec, w, precision=precision, hbm_budget=need), oracle.Model(spec, w)
    pot.reserve(*room)
    for _ in range(3):
        check(pot, orc, systems, precision)
    with pytest.raises(NNPError):
        Potential(spec, w, precision=precision, hbm_budget=need - 1).reserve(*room)


def test_pair_numbers_of_the_angular_blocks():
    """The (quotient, remainder) of the forward's triplet numbers from a float
    reciprocal off by up to two units in its last place, for every block of up to 512
    neighbours, and the circle's enumeration of the pairs of one species."""
    f = np.float32
    for cu in range(1, 513):
        t = np.arange(cu * 512, dtype=np.int64)
        inv0 = f(1) / f(cu)
        for inv in (inv0, inv0 * f(1 + 2 ** -22), inv0 * f(1 - 2 ** -22)):
            a = ((t.astype(f) + f(0.5)) * f(inv)).astype(np.int64)
            assert np.array_equal(a, t // cu)
    for n in range(2, 70):
        t = np.arange(n * (n - 1) // 2)
        a, b = t // n, t % n
        c = (a + b + 1) % n
        pairs = {(min(x, y), max(x, y)) for x, y in zip(b, c)}
        assert len(pairs) == t.size and np.all(b != c)
