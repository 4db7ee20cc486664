"""Persistent neighbour lists where their owner changes between calls: calls that the
caller captured into a CUDA graph, replayed after a force VJP or a call of another batch
layout on the same handle, and settings that order the AEV rows otherwise.

Every result is compared with a fresh evaluation (lists built at the cutoffs) and, once
per system, with the FP64 oracle: FP32 forces within 1e-4 of their RMS, energies within
1e-3 kcal/mol, as in the parity tests.
"""
import numpy as np
import pytest

import oracle
import synth
from tests._common import force_errors, model_for, to_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    return torch


class Case:
    """One system, its device arrays, and what a fresh evaluation gives for it."""

    def __init__(self, fresh, orc, s):
        import torch
        self.s, self.d = s, to_cuda(s)
        self.E = torch.zeros(1, dtype=torch.float64, device="cuda")
        self.F = torch.zeros((s.n_atoms, 3), dtype=torch.float32, device="cuda")
        E, F = fresh.energy_forces(self.d["coords"], self.d["species"], self.d["box"])
        self.ref = float(E.cpu()[0]), F.cpu().numpy().astype(np.float64)
        ref = orc.energy_forces(s.coords, s.species, s.box)
        self.f_rms = float(np.sqrt(np.mean(ref["forces"] ** 2)))
        rms, _ = force_errors(self.ref[1], ref["forces"])
        assert rms <= 1e-4 * self.f_rms and abs(self.ref[0] - ref["energy"]) <= 1e-3

    def call(self, pot):
        pot.energy_forces_into(self.d["coords"], self.d["species"], self.d["box"], None, self.E, self.F)

    def check(self, pot):
        assert pot.sync_status() == 0
        rms, _ = force_errors(self.F.cpu().numpy(), self.ref[1])
        assert rms <= 2e-5 * self.f_rms, rms
        assert abs(float(self.E.cpu()[0]) - self.ref[0]) <= 1e-6 * max(1.0, abs(self.ref[0]))
        self.F.zero_()
        self.E.zero_()

    def run(self, pot):
        self.call(pot)
        self.check(pot)


def captured(torch, fn):
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        fn()
    torch.cuda.synchronize()
    return g


def pair(kind, precision):
    from paper_2207_14276_gb300 import Potential
    spec, w = model_for(kind)
    fresh, kept = Potential(spec, w, precision=precision), Potential(spec, w, precision=precision)
    kept.set_skin(1.0)
    kept.reserve(1500, 2, 256, 160)   # the arena stays where it is, for the captured calls
    return fresh, kept, oracle.Model(spec, w)


@pytest.mark.parametrize("kind,precision", [("ani7x8", "fp32"), ("ani7", "fp32"), ("ani4", "fp32_simt")])
def test_captured_calls_find_the_lists_of_others(torch_cuda, kind, precision):
    torch = torch_cuda
    fresh, kept, orc = pair(kind, precision)
    if kind == "ani4":
        big, small = synth.water_box(300, 20.5, 7, seed=31), synth.water_box(100, 14.5, 5, seed=61)
    else:
        big, small = synth.solvated_solute(280, 40, 21.0, seed=6), synth.solvated_solute(100, 20, 15.5, seed=7)
    a, b = Case(fresh, orc, big), Case(fresh, orc, small)
    vjp = lambda c: kept.force_vjp_batch([c.d], [0.5], [torch.ones_like(c.F)])
    for c in (a, b, a, a):
        c.run(kept)
    graph = captured(torch, lambda: a.call(kept))   # with valid lists: none are built by itself
    builds = kept.list_stats()[0]
    graph.replay()
    a.check(kept)
    assert kept.list_stats()[0] == builds
    # a force VJP, of this system and of another one
    for c in (a, b):
        vjp(c)
        graph.replay()
        a.check(kept)
        graph.replay()
        a.check(kept)
    assert kept.list_stats()[0] == builds + 2
    # a call of another layout, and again after the replays have built their own lists
    for _ in range(2):
        b.run(kept)
        graph.replay()
        a.check(kept)
        b.run(kept)
        b.run(kept)
        graph.replay()
        a.check(kept)
    # the layout's own calls go on with the captured one's lists only if they are theirs
    a.run(kept)
    graph.replay()
    a.check(kept)
    # captured, but not run: the next call builds its lists
    b.run(kept)
    later = captured(torch, lambda: a.call(kept))
    a.run(kept)
    b.run(kept)
    later.replay()
    a.check(kept)


def test_captured_vjp_takes_the_lists_away(torch_cuda):
    torch = torch_cuda
    fresh, kept, orc = pair("ani7", "fp32")
    a = Case(fresh, orc, synth.solvated_solute(280, 40, 21.0, seed=6))
    v = torch.ones_like(a.F)
    kept.force_vjp_batch([a.d], [0.5], [v])   # its buffers exist now
    E, F, G = torch.zeros_like(a.E), torch.zeros_like(a.F), torch.zeros_like(a.F)
    W = torch.zeros(kept.n_weights, dtype=torch.float32, device="cuda")
    from paper_2207_14276_gb300 import _lib
    from paper_2207_14276_gb300.potential import _packed, _ptr, _stream_ptr
    arr = np.zeros(1, dtype=_lib.VJP_SYSTEM_DTYPE)
    arr["sys"] = np.frombuffer(_packed(a.d, {"energy": E, "forces": F}), dtype=_lib.SYSTEM_DTYPE)
    arr["dL_dE"], arr["dL_dF"], arr["dL_dcoords"] = 0.5, v.data_ptr(), G.data_ptr()
    graph = captured(torch, lambda: _lib.check(_lib.lib().nnp_force_vjp_batch(kept._h, 1, arr.ctypes.data, _ptr(W), _stream_ptr(None))))
    for _ in range(3):
        a.run(kept)
        a.run(kept)
        graph.replay()
    a.run(kept)


# settings that order the AEV rows otherwise, changed between calls that keep their lists
@pytest.mark.parametrize("kind,precision", [("ani7", "fp32"), ("ani7x8", "fp32_simt")])
def test_row_order_settings_between_kept_lists(torch_cuda, kind, precision):
    fresh, kept, orc = pair(kind, precision)
    a = Case(fresh, orc, synth.solvated_solute(280, 40, 21.0, seed=6))
    for sparse in (True, False, False, True, True, False, True):
        kept.set_sparse_rows(sparse)
        a.run(kept)
        a.run(kept)


def test_fused_first_layer_between_kept_lists(torch_cuda):
    torch = torch_cuda
    from paper_2207_14276_gb300 import Potential
    spec, w = model_for("ani4")
    fresh, kept = Potential(spec, w, precision="bf16"), Potential(spec, w, precision="bf16")
    kept.set_skin(1.0)
    d = to_cuda(synth.water_box(300, 20.5, 7, seed=31))
    E0, F0 = fresh.energy_forces(d["coords"], d["species"], d["box"])
    rms = float(F0.pow(2).mean().sqrt())
    for fused in (False, True, True, False, False, True):
        kept.set_fused_aev_l1(fused)
        for _ in range(2):
            E, F = kept.energy_forces(d["coords"], d["species"], d["box"])
            assert float((F - F0).pow(2).mean().sqrt()) <= 2e-2 * rms   # BF16 operands
            assert torch.isfinite(E).all()
