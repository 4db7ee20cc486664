"""Models and calls past the usual sizes, against the FP64 oracle.

Bounds, those of the parity tests: FP32 forces within 1e-4 of their RMS, energies within
1e-3 kcal/mol and within 1e-4 of sum_i |E_i|; BF16 forces within 2e-2 of their RMS (2^-9
relative per operand).
"""
import pytest

import oracle
import synth
from tests.test_gpu_shapes import check, model

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
